// C entry points that launch single kernels of csrc/strong.cu on the caller's data (host arrays), for
// tests/test_gpu_strong_kernels.py.
#include "../../paper_1007_4290_gb300/csrc/strong.cu"
#include "dev.cuh"

namespace {

// blocks of rows[bi] rows and P test vectors, one after the other in out
template <typename R>
int normals(int nblk, const int* rows, int P, unsigned m, unsigned seed, Cx<R>* out) {
  std::vector<int> info(8 * nblk, 0);
  std::vector<long long> off(nblk);
  long long o = 0;
  int most = 0;
  for (int b = 0; b < nblk; ++b) {
    info[8 * b + 5] = rows[b];
    off[b] = o;
    o += (long long)rows[b] * P;
    most = std::max(most, rows[b] * (P / 2));
  }
  Dev<int> di(info.size(), info.data());
  Dev<long long> doff(nblk, off.data());
  Dev<Cx<R>> d(o);
  if (!di.p || !doff.p || !d.p) return 2;
  FarArgs fa{};
  fa.nblk = nblk; fa.P = P; fa.seed = seed; fa.info = di.p; fa.soff = doff.p;
  strong_normals<R><<<dim3(nblk, (most + 127) / 128), 128>>>(fa, (int)m, d.p);
  return cudaDeviceSynchronize() == cudaSuccess && d.get(out) ? 0 : 4;
}

// the rank-R projection of one block F_a F_b^t (su x k, sw x k): its new factors Oa (su x R), Ob (sw x R)
template <typename R>
int far(int su, int sw, int k, int rank_cap, double eps, int shared, const Cx<R>* F, Cx<R>* O) {
  if (k > kKMax) return 1;
  const int P = std::min(kPMax, (rank_cap + kOversample + 1) / 2 * 2);
  const int info[8] = {0, 1, 0, 0, su, sw, 0, 1}, sz[2] = {su, sw}, rank[2] = {k, k};
  const long long soff[1] = {0}, gfo[2] = {0, (long long)su * k};
  Dev<int> di(8, info), dsz(2, sz), dr(2, rank);
  Dev<long long> ds(1, soff), dg(2, gfo);
  // (one offset table for input and output: the input's, with room for both)
  Dev<Cx<R>> dF((size_t)(su + sw) * k, F), dO((size_t)(su + sw) * std::max(k, rank_cap)), dS((size_t)(su + sw) * P);
  if (!di.p || !dsz.p || !dr.p || !ds.p || !dg.p || !dF.p || !dO.p || !dS.p || rank_cap > k) return 2;
  FarArgs fa{};
  fa.nblk = 1; fa.R = rank_cap; fa.P = P; fa.info = di.p; fa.soff = ds.p; fa.gfo = dg.p; fa.sz = dsz.p;
  fa.shared = shared;
  const size_t smem = shared ? (size_t)(su + sw) * P * sizeof(Cx<R>) : 0;
  cudaFuncSetAttribute(strong_far<R>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  strong_normals<R><<<dim3(1, (sw * (P / 2) + 127) / 128), 128>>>(fa, 3, dS.p);
  strong_far<R><<<1, kThreads, smem>>>(fa, (R)eps, dF.p, dr.p, dO.p, dS.p);
  if (cudaDeviceSynchronize() != cudaSuccess) return 4;
  cudaMemcpy(O, dO.p, sizeof(Cx<R>) * su * rank_cap, cudaMemcpyDeviceToHost);
  return cudaMemcpy(O + (size_t)su * rank_cap, dO.p + gfo[1], sizeof(Cx<R>) * sw * rank_cap, cudaMemcpyDeviceToHost) == cudaSuccess ? 0 : 5;
}

}  // namespace

ENTRY normals_f32(int nblk, const int* rows, int P, unsigned m, unsigned seed, Cx<float>* out) {
  return normals<float>(nblk, rows, P, m, seed, out);
}
ENTRY normals_f64(int nblk, const int* rows, int P, unsigned m, unsigned seed, Cx<double>* out) {
  return normals<double>(nblk, rows, P, m, seed, out);
}
ENTRY far_f32(int su, int sw, int k, int cap, double eps, int shared, const Cx<float>* F, Cx<float>* O) {
  return far<float>(su, sw, k, cap, eps, shared, F, O);
}
ENTRY far_f64(int su, int sw, int k, int cap, double eps, int shared, const Cx<double>* F, Cx<double>* O) {
  return far<double>(su, sw, k, cap, eps, shared, F, O);
}
