// C entry points that launch single kernels of csrc/setup.cu on the caller's data (host arrays), for tests/test_gpu_setup_kernels.py.
#include "../../paper_1007_4290_gb300/csrc/setup.cu"

#include "dev.cuh"

namespace {

// the truncated SVD of one core C (qa x qb, column-major): T_a (ld qcap, r_max columns), T_b, rank
template <typename R>
int svd(int qa, int qb, int qcap, int r_max, double eps, const Cx<R>* C, Cx<R>* Ta, Cx<R>* Tb, int* rank) {
  if (qa > qcap || qb > qcap) return 1;
  const int list[1] = {0}, qcols[2] = {qa, qb};
  Dev<int> dl(1, list), dq(2, qcols), dr(2);
  Dev<Cx<R>> dC((size_t)qcap * qcap), dT((size_t)2 * qcap * r_max);
  if (!dl.p || !dq.p || !dr.p || !dC.p || !dT.p) return 2;
  cudaMemcpy(dC.p, C, sizeof(Cx<R>) * qa * qb, cudaMemcpyHostToDevice);
  Geo g{};
  g.QCAP = qcap; g.r_max = r_max; g.list = dl.p;
  const SvdPlan<R> s(qcap, eps);
  if (s.smem > 227 * 1024) return 3;
  cudaFuncSetAttribute(svd_jacobi<R>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)s.smem);
  svd_jacobi<R><<<1, 1024, s.smem>>>(g, eps, dC.p, dq.p, dT.p, dr.p, s.entries, s.thr, s.rem);
  if (cudaDeviceSynchronize() != cudaSuccess) return 4;
  cudaMemcpy(Ta, dT.p, sizeof(Cx<R>) * qcap * r_max, cudaMemcpyDeviceToHost);
  cudaMemcpy(Tb, dT.p + (size_t)qcap * r_max, sizeof(Cx<R>) * qcap * r_max, cudaMemcpyDeviceToHost);
  return cudaMemcpy(rank, dr.p, sizeof(int), cudaMemcpyDeviceToHost) == cudaSuccess ? 0 : 5;
}

}  // namespace

ENTRY svd_f32(int qa, int qb, int qcap, int r_max, double eps, const Cx<float>* C, Cx<float>* Ta, Cx<float>* Tb, int* rank) {
  return svd<float>(qa, qb, qcap, r_max, eps, C, Ta, Tb, rank);
}
ENTRY svd_f64(int qa, int qb, int qcap, int r_max, double eps, const Cx<double>* C, Cx<double>* Ta, Cx<double>* Tb, int* rank) {
  return svd<double>(qa, qb, qcap, r_max, eps, C, Ta, Tb, rank);
}

namespace {

// the QR of one factor F (s x w, column-major), columns in shared memory (qsh) or in place: the kept Q
// columns (in F), R (row-major, ld w) and their number
template <typename R>
int qr(int s, int w, int qsh, Cx<R>* F, Cx<R>* Rm, int* qc) {
  if (w >= s) return 1;
  const int list[1] = {0}, sz[1] = {s}, cap[1] = {w}, rank[1] = {w};
  const long long off[1] = {0};
  Dev<int> dl(1, list), dsz(1, sz), dcap(1, cap), drk(1, rank), dq(1), dm(1);
  Dev<long long> doff(1, off);
  Dev<Cx<R>> dF((size_t)s * w, F), dR((size_t)w * w);
  if (!dl.p || !dsz.p || !dcap.p || !drk.p || !dq.p || !dm.p || !doff.p || !dF.p || !dR.p) return 2;
  Geo g{};
  g.cap_max = w; g.list = dl.p; g.sz = dsz.p; g.cap = dcap.p; g.gfo = doff.p; g.rbo = doff.p;
  const size_t base = qr_tables<R>(w), smem = base + (qsh ? (size_t)s * w * sizeof(Cx<R>) : 0);
  if (smem > 226 * 1024) return 3;
  cudaFuncSetAttribute(qr_mgs<R>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  qr_mgs<R><<<1, 1024, smem>>>(g, dF.p, drk.p, dR.p, dq.p, dm.p, qsh ? s * w : 0);
  if (cudaDeviceSynchronize() != cudaSuccess) return 4;
  return dF.get(F) && dR.get(Rm) && dq.get(qc) ? 0 : 5;
}

}  // namespace

ENTRY qr_f32(int s, int w, int qsh, Cx<float>* F, Cx<float>* Rm, int* qc) { return qr<float>(s, w, qsh, F, Rm, qc); }
ENTRY qr_f64(int s, int w, int qsh, Cx<double>* F, Cx<double>* Rm, int* qc) { return qr<double>(s, w, qsh, F, Rm, qc); }
