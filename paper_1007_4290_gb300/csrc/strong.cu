// Strong admissibility (Section 2.3, the strongly admissible case).  Clusters i, i' of one
// depth are well separated when the distance between them is at least their width, on
// the bisection tree of a layer: |i - i'| >= 2.  A strongly admissible H-matrix keeps the
// blocks of the interaction lists (well separated, parents not) in factorised form of
// rank at most R, and the neighbouring leaves (the near field) densely.
//
// The GPU builds T~_m in strong form from the weakly admissible inverse of the setup
// (setup.cu), in two exact-layout steps per layer:
//   projection: every well-separated block (u, w) lies inside one sibling block (a, b) of
//     the weak form, S(u, w) = F_a[rows u] F_b[rows w]^t; its rank-R approximation comes
//     from the randomized SVD (Halko, Martinsson and Tropp; the paper uses it for
//     F = H . H): Y = S Omega with P = R + 8 Gaussian test vectors, Q = orth(Y),
//     B = Q^* S, and the dominant right singular vectors P of B (one-sided Jacobi) give
//     S ~ S P P^*.  The near-field blocks (neighbouring
//     leaves) are formed densely;
//   expansion: the strong matrix is written back into the sibling-pair factor store
//     without approximation.  Inside a sibling block (a, b) the well-separated blocks
//     are, for every depth l below a, the three children (2c_a, 2c_b), (2c_a, 2c_b+1),
//     (2c_a+1, 2c_b+1) of the corner pair (c_a, c_b) (rightmost descendant of a, leftmost
//     of b at depth l-1), and the corner pair of leaves is dense, so F_a, F_b get the
//     columns [R per block | the corner block against the identity]: rank
//     3 R (L - depth(a)) + leaf.
// The next layer's S~_{m+1} and the sweeps read the expanded store, so both use the
// strongly admissible T~_m exactly.
#include <algorithm>
#include <cmath>
#include <vector>
#include "handle.h"

namespace {

constexpr int kThreads = 256;
constexpr int kOversample = 8;
constexpr int kPMax = 16;     // test vectors per block (R <= 8)
constexpr int kKMax = 56;     // rank of a weak block (r_max <= 56)

// Philox4x32-10 (Salmon, Moraes, Dror and Shaw, "Parallel random numbers: as easy as
// 1, 2, 3", SC 2011): ten rounds of the multiply-xor bijection keyed by a Weyl sequence.
__host__ __device__ inline void philox_round(uint32_t c[4], const uint32_t k[2]) {
  const uint64_t p0 = (uint64_t)0xD2511F53u * c[0];
  const uint64_t p1 = (uint64_t)0xCD9E8D57u * c[2];
  const uint32_t hi0 = (uint32_t)(p0 >> 32), lo0 = (uint32_t)p0;
  const uint32_t hi1 = (uint32_t)(p1 >> 32), lo1 = (uint32_t)p1;
  const uint32_t n0 = hi1 ^ c[1] ^ k[0], n2 = hi0 ^ c[3] ^ k[1];
  c[0] = n0; c[1] = lo1; c[2] = n2; c[3] = lo0;
}

}  // namespace

__host__ __device__ void hsw_philox4x32_10(const uint32_t ctr[4], const uint32_t key[2], uint32_t out[4]) {
  uint32_t c[4] = {ctr[0], ctr[1], ctr[2], ctr[3]};
  uint32_t k[2] = {key[0], key[1]};
  for (int r = 0; r < 10; ++r) {
    if (r > 0) { k[0] += 0x9E3779B9u; k[1] += 0xBB67AE85u; }
    philox_round(c, k);
  }
  for (int i = 0; i < 4; ++i) out[i] = c[i];
}

namespace {

// Two complex standard normals (real and imaginary parts independent N(0, 1)) from one
// Philox block, by the Box-Muller transform in FP64: the stored vectors are those of
// hsweep_rsvd_normals, rounded.
template <typename R>
__device__ inline void gauss2(uint32_t row, uint32_t pair, uint32_t blk, uint32_t m, uint32_t seed, Cx<R>& z0,
                              Cx<R>& z1) {
  const uint32_t ctr[4] = {row, pair, blk, m};
  const uint32_t key[2] = {seed, 0x5EEDu};
  uint32_t x[4];
  hsw_philox4x32_10(ctr, key, x);
  const double s = 2.3283064365386963e-10;   // 2^-32
  const double u0 = ((double)x[0] + 0.5) * s, u1 = (double)x[1] * s;
  const double u2 = ((double)x[2] + 0.5) * s, u3 = (double)x[3] * s;
  const double r0 = sqrt(-2.0 * log(u0)), r1 = sqrt(-2.0 * log(u2));
  double s0, c0, s1, c1;
  sincospi(2.0 * u1, &s0, &c0);
  sincospi(2.0 * u3, &s1, &c1);
  z0 = Cx<R>(R(r0 * c0), R(r0 * s0));
  z1 = Cx<R>(R(r1 * c1), R(r1 * s1));
}

struct FarArgs {
  int nblk, R, P;
  uint32_t seed;
  const int* info;          // [nblk][8]: a, b, ru0, rw0, su, sw, col, depth of (u, w)
  const long long* soff;    // [nblk] scratch offset (entries): Omega/Bt (sw x P), then Y/Q (su x P)
  const long long* gfo;     // factor offsets per node
  const int* sz;            // node sizes
  int shared;               // the scratch of every block fits in dynamic shared memory
};

// Omega of every block, complex Gaussian test vectors (sw x P, column-major) into its scratch: the
// FP64 logarithms and sines of the largest block take one SM longer than the block's products, so
// they are spread over the GPU first.
template <typename R>
__global__ void __launch_bounds__(128) strong_normals(FarArgs fa, int m, Cx<R>* __restrict__ scratch) {
  const int bi = blockIdx.x, sw = fa.info[8 * bi + 5], e = blockIdx.y * blockDim.x + threadIdx.x;
  if (e >= sw * (fa.P / 2)) return;
  const int row = e % sw, pr = e / sw;
  Cx<R> z0, z1;
  gauss2<R>((uint32_t)row, (uint32_t)pr, (uint32_t)bi, (uint32_t)m, fa.seed, z0, z1);
  Cx<R>* Om = scratch + fa.soff[bi];
  Om[(2 * pr) * sw + row] = z0;
  Om[(2 * pr + 1) * sw + row] = z1;
}

// Z[p][c] (ld kKMax) = sum_r F[r, c] v_p[r] (CONJ: conj(v_p[r])), c < k, p < np: a warp per
// column c and eight vectors
template <bool CONJ, typename R>
__device__ __forceinline__ void columns_dot(const Cx<R>* __restrict__ F, int ldf, int k, const Cx<R>* V, int rows, int np,
                                            Cx<R>* Z) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  const int pg = (np + 7) / 8;
  for (int e = warp; e < k * pg; e += nw) {
    const int c = e / pg, p0 = 8 * (e % pg);
    Cx<R> acc[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) acc[u] = Cx<R>(0, 0);
    for (int r = lane; r < rows; r += 32) {
      const Cx<R> f = F[(long long)c * ldf + r];
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const Cx<R> v = V[min(p0 + u, np - 1) * rows + r];
        if (CONJ) cfma_conj(acc[u], v, f);
        else cfma(acc[u], v, f);
      }
    }
    int u;
    bool first;
    scatter_sum<R, 8, 32, 1>(acc, lane, u, first);
    if (first && p0 + u < np) Z[(p0 + u) * kKMax + c] = acc[0];
  }
}

// put(r, p, sum_c F[r, c] Z[p][c]) for r < rows, p < np: a thread per row and four vectors
template <typename R, typename Put>
__device__ __forceinline__ void rows_times(const Cx<R>* __restrict__ F, int ldf, int k, const Cx<R>* Z, int rows, int np,
                                           Put put) {
  const int pg = (np + 3) / 4;
  for (int e = threadIdx.x; e < rows * pg; e += blockDim.x) {
    const int r = e % rows, p0 = 4 * (e / rows);
    Cx<R> acc[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) acc[u] = Cx<R>(0, 0);
#pragma unroll 4
    for (int c = 0; c < k; ++c) {
      const Cx<R> f = F[(long long)c * ldf + r];
#pragma unroll
      for (int u = 0; u < 4; ++u) cfma(acc[u], f, Z[min(p0 + u, np - 1) * kKMax + c]);
    }
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (p0 + u < np) put(r, p0 + u, acc[u]);
  }
}

// One CTA per well-separated block: randomized rank-R projection, written into the
// expanded factors of the sibling pair (a, b) that contains it.  The basis of the sampled
// range comes from two rounds of right-looking Gram-Schmidt (a warp per later column, one
// barrier a step); the dominant right singular vectors of B = Q^* S from one-sided Jacobi on
// the columns of B^t (a warp per pair); and the left factor from the product of S with them,
// so that the result is the projection S P P^* whatever the basis.  What bounds it is the
// latency of these short chains; with classical Gram-Schmidt (a block-wide sum per inner
// product) and FP64 Jacobi on the Gram matrix by one warp a layer at n = 255 took 931 us, now 71.
template <typename R>
__global__ void __launch_bounds__(kThreads) strong_far(FarArgs fa, R eps, const Cx<R>* __restrict__ F,
                                                       const int* __restrict__ rank, Cx<R>* __restrict__ Fout,
                                                       Cx<R>* __restrict__ scratch) {
  extern __shared__ __align__(16) unsigned char dyn[];
  __shared__ Cx<R> Z[kKMax * kPMax];
  __shared__ R cur[kPMax], org[kPMax], sig[kPMax];
  __shared__ int kept[kPMax], order[kPMax];
  __shared__ int s_rot, s_gg, s_t, s_keep;

  const int bi = blockIdx.x;
  const int* inf = fa.info + 8 * bi;
  const int a = inf[0], b = inf[1], ru0 = inf[2], rw0 = inf[3], su = inf[4], sw = inf[5], col = inf[6];
  const int k = rank[a];
  if (k <= 0) return;
  const int P = fa.P, tid = threadIdx.x;
  const int warp = tid >> 5, lane = tid & 31, nw = kThreads / 32;
  const int lda = fa.sz[a], ldb = fa.sz[b];
  const Cx<R>* Fa = F + fa.gfo[a] + ru0;
  const Cx<R>* Fb = F + fa.gfo[b] + rw0;
  Cx<R>* Om = fa.shared ? reinterpret_cast<Cx<R>*>(dyn) : scratch + fa.soff[bi];   // sw x P (Omega, later Bt)
  Cx<R>* Y = Om + sw * P;                                                            // su x P (Y, then Q)

  if (fa.shared) {
    const Cx<R>* src = scratch + fa.soff[bi];
    for (int e = tid; e < sw * P; e += blockDim.x) Om[e] = src[e];
    __syncthreads();
  }
  // Y = S Omega = F_a[rows u] (F_b[rows w]^t Omega)
  columns_dot<false>(Fb, ldb, k, Om, sw, P, Z);
  __syncthreads();
  rows_times(Fa, lda, k, Z, su, P, [&](int r, int p, Cx<R> v) { Y[p * su + r] = v; });
  __syncthreads();
  // Q = orth(Y), dependent columns dropped; the second round restores the orthogonality the
  // first one lost on columns with small remainders
  const R keep_tol = sizeof(R) == 4 ? R(1e-5) : R(1e-12);
  int q = 0;
  for (int round = 0; round < 2; ++round) {
    const int nc = round == 0 ? P : q;
    for (int j = warp; j < nc; j += nw) {
      const Cx<R>* y = Y + (round == 0 ? j : kept[j]) * su;
      R acc = 0;
      for (int r = lane; r < su; r += 32) acc += abs2(y[r]);
      for (int o = 16; o; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
      if (lane == 0) cur[j] = org[j] = acc;
    }
    __syncthreads();
    int qn = 0;
    for (int j = 0; j < nc; ++j) {
      const R nr = cur[j];
      const bool keep = round == 1 || (nr > keep_tol * keep_tol * org[j] && nr > R(0));
      const int src = round == 0 ? j : kept[j];
      if (keep) {
        const Cx<R>* yj = Y + src * su;
        const R inv = rcp_any(nr);
        for (int l = j + 1 + warp; l < nc; l += nw) {
          Cx<R>* yl = Y + (round == 0 ? l : kept[l]) * su;
          Cx<R> d(0, 0);
          for (int r = lane; r < su; r += 32) cfma_conj(d, yj[r], yl[r]);
          for (int o = 16; o; o >>= 1) d += shfl_xor(d, o);
          const Cx<R> be = -(inv * d);
          R acc = 0;
          for (int r = lane; r < su; r += 32) {
            Cx<R> v = yl[r];
            cfma(v, be, yj[r]);
            yl[r] = v;
            acc += abs2(v);
          }
          for (int o = 16; o; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
          if (lane == 0) cur[l] = acc;
        }
      }
      __syncthreads();
      if (keep) {
        if (round == 0 && tid == 0) kept[qn] = j;
        ++qn;
      }
    }
    q = qn;
    __syncthreads();
    // normalise (after the first round, the kept columns' norms again)
    for (int j = warp; j < q; j += nw) {
      Cx<R>* y = Y + kept[j] * su;
      const R rs = rsqrt_any(cur[round == 0 ? kept[j] : j]);
      for (int r = lane; r < su; r += 32) y[r] = rs * y[r];
    }
    __syncthreads();
  }
  if (q == 0) return;
  // the kept columns side by side (a column never lies before its place)
  for (int j = 0; j < q; ++j) {
    const int src = kept[j];
    if (src != j)
      for (int r = tid; r < su; r += blockDim.x) Y[j * su + r] = Y[src * su + r];
    __syncthreads();
  }
  // Bt = (Q^* S)^t = F_b[rows w] (F_a[rows u]^t conj(Q))  (sw x q), over Omega
  columns_dot<true>(Fa, lda, k, Y, su, q, Z);
  __syncthreads();
  rows_times(Fb, ldb, k, Z, sw, q, [&](int r, int p, Cx<R> v) { Om[p * sw + r] = v; });
  __syncthreads();
  // one-sided Jacobi on the q columns of Bt, scaled by the largest: Bt W = P Sigma
  for (int j = warp; j < q; j += nw) {
    R acc = 0;
    for (int r = lane; r < sw; r += 32) acc += abs2(Om[j * sw + r]);
    for (int o = 16; o; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (lane == 0) sig[j] = acc;
  }
  __syncthreads();
  R scale2 = 0;
  for (int j = 0; j < q; ++j) scale2 = fmax(scale2, sig[j]);
  if (!(scale2 > R(0))) return;
  const R iscale = rsqrt_any(scale2);
  const R floor2 = sizeof(R) == 4 ? R(1e-14) : R(1e-28);
  const float tol2 = sizeof(R) == 4 ? 1.6e-13f : 1e-30f, quad = sizeof(R) == 4 ? 1e-8f : 1e-16f;
  __syncthreads();
  for (int e = tid; e < sw * q; e += blockDim.x) Om[e] = iscale * Om[e];
  const int me = q + (q & 1);
  for (int sweep = 0; sweep < 30; ++sweep) {
    __syncthreads();
    if (tid == 0) s_rot = s_gg = s_t = 0;
    __syncthreads();
    for (int round = 0; round < me - 1; ++round) {
      for (int pr = warp; pr < me / 2; pr += nw) {
        const int p1 = me - 1 - pr;
        const int ip = pr == 0 ? 0 : (pr - 1 + round) % (me - 1) + 1, iq = (p1 - 1 + round) % (me - 1) + 1;
        if (ip >= q || iq >= q) continue;
        Cx<R>* cp = Om + min(ip, iq) * sw;
        Cx<R>* cq = Om + max(ip, iq) * sw;
        R al = 0, be = 0;
        Cx<R> ga(0, 0);
        for (int r = lane; r < sw; r += 32) {
          const Cx<R> x = cp[r], y = cq[r];
          al += abs2(x);
          be += abs2(y);
          cfma_conj(ga, x, y);
        }
        for (int o = 16; o; o >>= 1) {
          al += __shfl_xor_sync(0xffffffffu, al, o);
          be += __shfl_xor_sync(0xffffffffu, be, o);
          ga += shfl_xor(ga, o);
        }
        if (!(al >= floor2 && be >= floor2)) continue;
        JacobiRotation<R> rot;
        if (!rot.needed(al, be, ga, tol2)) continue;
        rot.angle(al, be);
        if (lane == 0) {
          if (rot.gg > quad) {
            s_rot = 1;
          } else {
            atomicMax(&s_gg, __float_as_int(rot.gg));
            atomicMax(&s_t, __float_as_int(fabsf(rot.t)));
          }
        }
        for (int r = lane; r < sw; r += 32) {
          const Cx<R> x = cp[r], y = cq[r];
          Cx<R> nx = rot.cs * x, ny = rot.cs * y;
          cfma(nx, -conj(rot.sne), y);
          cfma(ny, rot.sne, x);
          cp[r] = nx;
          cq[r] = ny;
        }
      }
      __syncthreads();
    }
    if (s_rot == 0 && rotations_done(__int_as_float(s_gg), __int_as_float(s_t), tol2)) break;
  }
  for (int j = warp; j < q; j += nw) {
    R acc = 0;
    for (int r = lane; r < sw; r += 32) acc += abs2(Om[j * sw + r]);
    for (int o = 16; o; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (lane == 0) sig[j] = acc;
  }
  if (tid == 0) s_keep = 0;
  __syncthreads();
  if (tid < q) {
    int rk = 0;
    R smax = 0;
    for (int l = 0; l < q; ++l) {
      rk += (sig[l] > sig[tid] || (sig[l] == sig[tid] && l < tid)) ? 1 : 0;
      smax = fmax(smax, sig[l]);
    }
    order[rk] = tid;
    const R floor_rel = sizeof(R) == 4 ? R(1e-12) : R(1e-27);     // clear of the columns left unrotated
    if (rk < fa.R && sig[tid] > smax * fmax(eps * eps, floor_rel)) atomicMax(&s_keep, rk + 1);
  }
  __syncthreads();
  const int keep = s_keep;
  // F'_b[rows w] = P Sigma^(1/2), F'_a[rows u] = S conj(P) Sigma^(-1/2); column i of Om is
  // P sigma / scale, sigma = scale sqrt(sig)
  const R scale = scale2 * iscale;
  Cx<R>* Oa = Fout + fa.gfo[a] + ru0;
  Cx<R>* Ob = Fout + fa.gfo[b] + rw0;
  for (int e = tid; e < sw * keep; e += blockDim.x) {
    const int r = e % sw, i = e / sw;
    const R sg = sqrt(sig[order[i]]);
    Ob[(long long)(col + i) * ldb + r] = sqrt(scale / sg) * Om[order[i] * sw + r];
  }
  __syncthreads();
  for (int i = 0; i < keep; ++i) columns_dot<true>(Fb, ldb, k, Om + order[i] * sw, sw, 1, Z + i * kKMax);
  __syncthreads();
  rows_times(Fa, lda, k, Z, su, keep, [&](int r, int i, Cx<R> v) {
    const R sg = sqrt(sig[order[i]]);
    Oa[(long long)(col + i) * lda + r] = (R(1) / (sg * sqrt(scale * sg))) * v;
  });
}

struct NearArgs {
  const int* info;          // [npairs][6]: a, b, ca0 (rows of c_a within a), na, nb, col
  const long long* gfo;
  const int* sz;
};

// One CTA per sibling pair (a, b): the dense near-field block of its corner leaves
// D = F_a[rows c_a] F_b[rows c_b]^t, written as the columns [D | I] of the expansion.
template <typename R>
__global__ void __launch_bounds__(128) strong_near(NearArgs na, const Cx<R>* __restrict__ F, const int* __restrict__ rank,
                                                   Cx<R>* __restrict__ Fout) {
  const int* inf = na.info + 6 * blockIdx.x;
  const int a = inf[0], b = inf[1], ca0 = inf[2], nA = inf[3], nB = inf[4], col = inf[5];
  const int k = rank[a];
  const int lda = na.sz[a], ldb = na.sz[b];
  const Cx<R>* Fa = F + na.gfo[a] + ca0;
  const Cx<R>* Fb = F + na.gfo[b];
  Cx<R>* Oa = Fout + na.gfo[a] + ca0;
  Cx<R>* Ob = Fout + na.gfo[b];
  for (int e = threadIdx.x; e < nA * nB; e += blockDim.x) {
    const int i = e % nA, c = e / nA;
    Cx<R> acc(0, 0);
    for (int t = 0; t < k; ++t) cfma(acc, Fa[(long long)t * lda + i], Fb[(long long)t * ldb + c]);
    Oa[(long long)(col + c) * lda + i] = acc;
  }
  for (int e = threadIdx.x; e < nB * nB; e += blockDim.x) {
    const int i = e % nB, c = e / nB;
    Ob[(long long)(col + c) * ldb + i] = Cx<R>(i == c ? R(1) : R(0), R(0));
  }
}

int depth_of_host(int v) { int d = 0; while (v > 1) { v >>= 1; ++d; } return d; }

}  // namespace

struct StrongWork {
  int nfar = 0, nnear = 0, P = 0;
  int ngrid = 0;                // CTAs of strong_normals per block
  int* d_far = nullptr;
  long long* d_soff = nullptr;
  int* d_near = nullptr;
  int* d_rank = nullptr;        // expanded rank per node
  void* scratch = nullptr;
  size_t smem = 0;              // dynamic shared memory for the largest block's vectors (0: scratch)
};

int hsw_strong_expansion_rank(int R, int L, int leaf) { return 3 * R * (L > 0 ? L - 1 : 0) + leaf; }

// The strong layout of one layer: far records {a, b, ru0, rw0, su, sw, col, l} (the block
// (u, w) of depth l inside the sibling pair (a, b), rows ru0.. of a and rw0.. of b, columns
// col..col+R of the expanded factors), near records {a, b, ca0, na, nb, col} (the corner
// leaves), and the expanded rank of every node.
static void strong_plan(const Tree& t, int R, std::vector<int>& far, std::vector<int>& near,
                        std::vector<int>& nrank) {
  const int L = t.L;
  far.clear(); near.clear();
  nrank.assign(t.nnodes, 0);
  // the sibling pairs (a, b) and, inside each, the corner chain down to the leaves
  for (int av = 2; av < t.nnodes; av += 2) {
    const int bv = av + 1, la = depth_of_host(av);
    int ca = av, cb = bv;      // corner pair at depth l - 1
    for (int l = la + 1; l <= L; ++l) {
      const int us[3] = {2 * ca, 2 * ca, 2 * ca + 1};
      const int ws[3] = {2 * cb, 2 * cb + 1, 2 * cb + 1};
      for (int tt = 0; tt < 3; ++tt) {
        const int u = us[tt], w = ws[tt];
        const int rec[8] = {av, bv, t.lo[u] - t.lo[av], t.lo[w] - t.lo[bv], t.sz[u], t.sz[w],
                            R * (3 * (l - la - 1) + tt), l};
        far.insert(far.end(), rec, rec + 8);
      }
      ca = 2 * ca + 1;
      cb = 2 * cb;
    }
    // ca, cb are now the corner leaves
    const int col = 3 * R * (L - la);
    const int rec[6] = {av, bv, t.lo[ca] - t.lo[av], t.sz[ca], t.sz[cb], col};
    near.insert(near.end(), rec, rec + 6);
    nrank[av] = nrank[bv] = col + t.sz[cb];
  }
}

static int strong_prepare(hsweep_s* h, size_t es) {
  StrongWork* s = new (std::nothrow) StrongWork();
  if (!s) return HSWEEP_ERR_OOM;
  h->stw = s;
  const Tree& t = h->tree;
  s->P = std::min(kPMax, (h->strong_R + kOversample + 1) / 2 * 2);
  std::vector<int> far, near, nrank;
  strong_plan(t, h->strong_R, far, near, nrank);
  for (int v = 2; v < h->nnodes; ++v)
    if (nrank[v] > h->r_max) return HSWEEP_ERR_ARG;
  std::vector<long long> soff;
  long long so = 0;
  size_t most = 0;
  for (size_t i = 0; i < far.size(); i += 8) {
    most = std::max(most, (size_t)(far[i + 4] + far[i + 5]) * s->P * es);
    soff.push_back(so);
    s->ngrid = std::max(s->ngrid, (far[i + 5] * (s->P / 2) + 127) / 128);
    so += (long long)(far[i + 4] + far[i + 5]) * s->P;
  }
  // (Z and the tables take up to 15 KB of static shared memory beside it)
  s->smem = most <= 160 * 1024 ? most : 0;
  s->nfar = (int)soff.size();
  s->nnear = (int)(near.size() / 6);
  int rc;
  if ((rc = hsw_alloc(h, (void**)&s->d_far, std::max<size_t>(1, far.size()) * sizeof(int)))) return rc;
  if ((rc = hsw_alloc(h, (void**)&s->d_soff, std::max<size_t>(1, soff.size()) * sizeof(long long)))) return rc;
  if ((rc = hsw_alloc(h, (void**)&s->d_near, std::max<size_t>(1, near.size()) * sizeof(int)))) return rc;
  if ((rc = hsw_alloc(h, (void**)&s->d_rank, h->nnodes * sizeof(int)))) return rc;
  if ((rc = hsw_alloc(h, &s->scratch, (size_t)std::max(1LL, so) * es))) return rc;
  if (!far.empty())
    HSW_CUDA(cudaMemcpyAsync(s->d_far, far.data(), far.size() * sizeof(int), cudaMemcpyHostToDevice, h->stream));
  if (!soff.empty())
    HSW_CUDA(cudaMemcpyAsync(s->d_soff, soff.data(), soff.size() * sizeof(long long), cudaMemcpyHostToDevice, h->stream));
  if (!near.empty())
    HSW_CUDA(cudaMemcpyAsync(s->d_near, near.data(), near.size() * sizeof(int), cudaMemcpyHostToDevice, h->stream));
  HSW_CUDA(cudaMemcpyAsync(s->d_rank, nrank.data(), h->nnodes * sizeof(int), cudaMemcpyHostToDevice, h->stream));
  // the host vectors go out of scope: wait for the copies
  HSW_CUDA(cudaStreamSynchronize(h->stream));
  return HSWEEP_OK;
}

void hsw_strong_free(hsweep_s* h) {
  if (!h->stw) return;
  StrongWork* s = h->stw;
  void* ptrs[] = {s->d_far, s->d_soff, s->d_near, s->d_rank, s->scratch};
  for (void* p : ptrs) hsw_release(h, p);
  delete s;
  h->stw = nullptr;
}

template <typename R>
static int project_impl(hsweep_s* h, int m, const Cx<R>* G_F, int* G_rank, Cx<R>* G_F2, const long long* d_gfo,
                        long long gf_entries) {
  if (!h->stw) {
    int rc = strong_prepare(h, sizeof(Cx<R>));
    if (rc) return rc;
  }
  StrongWork* s = h->stw;
  cudaStream_t st = h->stream;
  HSW_CUDA(cudaMemsetAsync(G_F2, 0, (size_t)gf_entries * sizeof(Cx<R>), st));
  if (s->nfar > 0) {
    FarArgs fa;
    fa.nblk = s->nfar; fa.R = h->strong_R; fa.P = s->P; fa.seed = h->opt.rsvd_seed;
    fa.info = s->d_far; fa.soff = s->d_soff; fa.gfo = d_gfo; fa.sz = h->d_sz;
    fa.shared = s->smem > 0;
    if (s->smem > 0)
      HSW_CUDA(cudaFuncSetAttribute(strong_far<R>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)s->smem));
    strong_normals<R><<<dim3(s->nfar, s->ngrid), 128, 0, st>>>(fa, m, (Cx<R>*)s->scratch);
    strong_far<R><<<s->nfar, kThreads, s->smem, st>>>(fa, (R)h->eps_H, G_F, G_rank, G_F2, (Cx<R>*)s->scratch);
    h->nlaunch += 2;
  }
  if (s->nnear > 0) {
    NearArgs na;
    na.info = s->d_near; na.gfo = d_gfo; na.sz = h->d_sz;
    strong_near<R><<<s->nnear, 128, 0, st>>>(na, G_F, G_rank, G_F2);
    h->nlaunch += 1;
  }
  HSW_CUDA(cudaMemcpyAsync(G_rank, s->d_rank, h->nnodes * sizeof(int), cudaMemcpyDeviceToDevice, st));
  HSW_CUDA(cudaGetLastError());
  return HSWEEP_OK;
}

int hsw_strong_project(hsweep_s* h, int m, const void* G_F, int* G_rank, void* G_F2, const long long* d_gfo,
                       long long gf_entries) {
  if (h->prec == HSWEEP_FP64)
    return project_impl<double>(h, m, (const c128*)G_F, G_rank, (c128*)G_F2, d_gfo, gf_entries);
  return project_impl<float>(h, m, (const c64*)G_F, G_rank, (c64*)G_F2, d_gfo, gf_entries);
}

extern "C" int hsweep_strong_plan(int n, int leaf, int R, int* nfar, int* nnear, int* far, int* near, int* ranks) {
  if (n < 3 || n > 32767 || leaf < 2 || leaf > 8 || R < 1 || R > 8 || !nfar || !nnear) return HSWEEP_ERR_ARG;
  Tree t;
  t.build(n, leaf);
  std::vector<int> fv, nv, rk;
  strong_plan(t, R, fv, nv, rk);
  *nfar = (int)(fv.size() / 8);
  *nnear = (int)(nv.size() / 6);
  if (far) std::copy(fv.begin(), fv.end(), far);
  if (near) std::copy(nv.begin(), nv.end(), near);
  if (ranks) std::copy(rk.begin(), rk.end(), ranks);
  return HSWEEP_OK;
}

extern "C" int hsweep_rsvd_normals(uint32_t blk, uint32_t m, uint32_t seed, int rows, int P, double* out) {
  if (rows < 0 || P < 2 || (P & 1) || (rows > 0 && !out)) return HSWEEP_ERR_ARG;
  const double s = 2.3283064365386963e-10, two_pi = 6.283185307179586476925286766559;
  for (int pr = 0; pr < P / 2; ++pr)
    for (int row = 0; row < rows; ++row) {
      const uint32_t ctr[4] = {(uint32_t)row, (uint32_t)pr, blk, m};
      const uint32_t key[2] = {seed, 0x5EEDu};
      uint32_t x[4];
      hsw_philox4x32_10(ctr, key, x);
      const double u0 = ((double)x[0] + 0.5) * s, u1 = (double)x[1] * s;
      const double u2 = ((double)x[2] + 0.5) * s, u3 = (double)x[3] * s;
      const double r0 = std::sqrt(-2.0 * std::log(u0)), r1 = std::sqrt(-2.0 * std::log(u2));
      double* z0 = out + 2 * ((long long)(2 * pr) * rows + row);
      double* z1 = out + 2 * ((long long)(2 * pr + 1) * rows + row);
      z0[0] = r0 * std::cos(two_pi * u1); z0[1] = r0 * std::sin(two_pi * u1);
      z1[0] = r1 * std::cos(two_pi * u3); z1[1] = r1 * std::sin(two_pi * u3);
    }
  return HSWEEP_OK;
}

extern "C" int hsweep_philox4x32_10(const uint32_t* ctr, const uint32_t* key, uint32_t* out) {
  if (!ctr || !key || !out) return HSWEEP_ERR_ARG;
  hsw_philox4x32_10(ctr, key, out);
  return HSWEEP_OK;
}
