// The setup sweep of Algorithm 2.5 on the GPU: for m = 1..n
//   S~_m = A_mm - A_{m,m-1} T~_{m-1} A_{m-1,m}   (hdiagmul + hsub; Section 2.3)
//   T~_m = hinv(S~_m)
// with every matrix a weakly admissible H-matrix in symmetric storage (siblings a, b:
// block (a, b) = F_a F_b^t, block (b, a) = F_b F_a^t; dense leaves).
//
// hinv is organised level by level, bottom-up, instead of the paper's depth-first
// 2 x 2 recursion; both give the same inverse before truncation.  For a node t with
// children a, b and S(a, b) = U V^t:
//     S_t = diag(S_a, S_b) + P C P^t,  P = diag(U, V),  C = [[0, I], [I, 0]],
// so by the Woodbury identity, with G_a = S_a^{-1} and G_b = S_b^{-1} already built,
//     Y = diag(G_a U, G_b V),  M = [[U^t Y_a, I], [I, V^t Y_b]]^{-1},
//     S_t^{-1} = diag(G_a, G_b) - Y M Y^t.
// The new off-diagonal block is -Y_a M12 Y_b^t; the diagonal corrections -Y_a M11 Y_a^t
// and -Y_b M22 Y_b^t are rank-k updates of every block below a and b ("hadd" with a
// factorised term).  All nodes of one depth are processed by the same launches.
// Recompression ("Matrix addition": QR of both factors, SVD of the small core,
// truncation at eps_H relative to the block's largest singular value, at most r_max
// terms) runs once per layer, after the last depth, on every block whose final core fits
// the SVD's shared memory: appended columns accumulate (up to depth x (r_max + 1) of
// them), the untruncated factors feed the products of the higher depths, and each block
// is truncated once, in its final form.  Blocks whose core would not fit (large blocks
// in complex128) are recompressed after every depth that changed them.  A small block whose factors have at least as
// many columns as rows takes the dense path: its core is the block itself, C = F_a F_b^t,
// and its new factors come straight from the SVD of C (no QR).  QR is modified
// Gram-Schmidt, repeated for columns that lose most of themselves; the SVD is a column-pivoted Gram-Schmidt down to
// the numerical rank followed by one-sided (Hestenes) Jacobi on what remains.
// The leaf inverses are computed in FP64 with partial pivoting in both precisions.
#include <algorithm>
#include <cfloat>
#include <cmath>
#include <utility>
#include "handle.h"

namespace {

constexpr int kBlk = 256;

// Dense path of the recompression in complex64: up to this many rows the pivoted Gram-Schmidt
// of the block itself (svd_jacobi: one barrier for each of the block's 20 to 40 significant
// columns) is shorter than the QR of its factors (one for each of up to 98 columns).  A
// 128 x 128 core is 131 KB of shared memory.  In complex128 the QR is the cheaper.
constexpr int kDenseRows = 128;

template <typename R> struct Tiny;
template <> struct Tiny<double> {
  static constexpr double dep = 1e-13;    // Gram-Schmidt: dependent-column threshold
  static constexpr float jac2 = 1e-30f;   // Jacobi: orthogonality tolerance 1e-15 (about 8 ulp), squared
  static constexpr double neg = 1e-28;    // Jacobi: squared norm of a rounding-noise column
                                          // (normalised: below 1e-14 of the largest column)
  static constexpr float quad = 1e-16f;   // Jacobi: squared cosine from which one more sweep
                                          // is needed (the convergence is quadratic: a sweep
                                          // whose cosines were below 1e-8 leaves 1e-16)
};
template <> struct Tiny<float> {
  static constexpr float dep = 2e-6f;
  static constexpr float jac2 = 1.6e-13f; // (4e-7)^2, about 7 ulp: tighter only rotates rounding noise
  static constexpr float neg = 1e-14f;    // below 1e-7 of the largest column: FP32 noise
  static constexpr float quad = 1e-8f;
};

// Thresholds and shared memory of svd_jacobi for cores of at most qcap x qcap.
//   thr: columns with smaller squared norms (relative to the largest column's) are not rotated.
//   rem: the pivoted Gram-Schmidt ends when the squares of all that is left sum to this.
// Both are fractions of the truncation threshold eps.  A quarter and a hundredth in complex64: what is
// left holds no singular value above eps / 2, or two thirds of eps where the Gram matrix shows it to be
// noise (a sixteenth for rem takes two columns more at the top of n = 255 in the strong format, 286 for
// 266 ms a setup; each column against eps / 4, without a bound on their sum, 252 ms, but 128 aligned
// ones hold a value of 2.8 eps).
template <typename R>
struct SvdPlan {
  int entries;       // of the core
  size_t smem;       // the core, two rows of R, norms, singular values and index tables
  R thr;
  float rem;
  SvdPlan(int qcap, double eps) {
    entries = qcap * qcap;
    smem = ((size_t)entries + 2 * qcap) * sizeof(Cx<R>) + (size_t)(3 * qcap + 1) * sizeof(R) + (size_t)2 * qcap * sizeof(int) + 16;
    thr = (R)std::max((double)Tiny<R>::neg, (sizeof(R) == 4 ? 0.01 : 0.0025) * eps * eps);
    rem = (float)((sizeof(R) == 4 ? 0.25 : 0.0025) * eps * eps);
  }
};

template <typename R> __device__ __forceinline__ R warp_sum_r(R v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// 1 / a, by the Newton reciprocal where |a|^2 is well inside FP32's range
__device__ __forceinline__ c128 cinv_fast(c128 a) {
  const double d = abs2(a);
  const double s = (d > 1e-30 && d < 1e30) ? rcp_of(d) : 1.0 / d;
  return c128(a.re * s, -a.im * s);
}

// Programmatic dependent launch: a kernel lets its successor's CTAs start (they wait here for
// its end), so that the launch latency between the layer's forty short kernels is hidden
// (about 1 us each; no effect on kernels launched without the attribute).
__device__ __forceinline__ void pdl_begin() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
}
template <typename... KA, typename... A>
static cudaError_t pdl_launch(void (*kern)(KA...), dim3 grid, int block, size_t smem, cudaStream_t st, A... args) {
  cudaLaunchConfig_t lc = {};
  lc.gridDim = grid;
  lc.blockDim = dim3(block);
  lc.dynamicSmemBytes = smem;
  lc.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  lc.attrs = at;
  lc.numAttrs = 1;
  return cudaLaunchKernelEx(&lc, kern, KA(args)...);
}

struct Geo {          // tree and buffer geometry passed by value to every kernel
  int n, L, leaf, nnodes, r_max, KCAP, WCAP, QCAP;
  int cap_max;             // the largest cap
  int dense_max;           // blocks of at most so many rows take the dense path at any rank
  const int* lo;
  const int* sz;
  const int* rowleaf;      // [n] leaf node of each row
  const long long* sfo;    // S factor offsets (capacity KCAP per node)
  const long long* gfo;    // G factor offsets (capacity cap[v] columns per node)
  const int* cap;          // column capacity of every node's G factor
  const long long* qro;    // offsets of the reductions Qr (cap[v] x KCAP per node)
  const long long* rbo;    // offsets of the R factors (min(sz, cap) x cap, row-major, ld cap)
  const int* list;         // recompression kernels: the nodes (or left siblings) to process
};

__device__ __forceinline__ int depth_of(int v) { return 31 - __clz(v); }

// ---------------------------------------------------------------------------------
// S~_m, one launch: blocks 0 .. nleaves - 1 (of slice 0) form a leaf A_mm[leaf] - D T_leaf D
// and invert it, FP64 Gauss-Jordan with partial pivoting in both precisions (a serial chain
// of FP64 instructions, 17 us, with the factors beside it; 35 us in three launches before); the others form the factors
// [-D F_a, a e_last] / [D F_b, e_first] of node v = 2 + blockIdx.x - nleaves, in gridDim.y slices.
template <typename R>
__global__ void __launch_bounds__(kBlk) schur_layer(Geo g, int m, const c128* __restrict__ diag,
                                                    const c128* __restrict__ east, const c128* __restrict__ north,
                                                    const Cx<R>* __restrict__ Tprev, const long long* __restrict__ toff,
                                                    const int* __restrict__ trank, Cx<R>* __restrict__ S_F,
                                                    int* __restrict__ S_rank, Cx<R>* __restrict__ G_leaf,
                                                    int* __restrict__ G_rank, int* status) {
  pdl_begin();
  const int nleaves = 1 << g.L;
  if ((int)blockIdx.x >= nleaves) {
    const int v = 2 + (int)blockIdx.x - nleaves;
    const int lo = g.lo[v], s = g.sz[v];
    const bool left = (v & 1) == 0;
    const int r0 = Tprev ? trank[v] : 0;
    const int k = r0 + 1;
    Cx<R>* dst = S_F + g.sfo[v];
    const int edge = g.lo[v | 1];     // the coupling edge joins rows edge-1 and edge
    for (int e = blockIdx.y * blockDim.x + threadIdx.x; e < s * k; e += gridDim.y * blockDim.x) {
      const int i = e % s, col = e / s;
      Cx<R> val(0, 0);
      if (col < r0) {
        Cx<R> dv = cvt<R>(north[(long long)m * g.n + lo + i]);
        val = dv * Tprev[toff[v] + (long long)col * s + i];
        if (left) val = -val;
      } else if (i == (left ? s - 1 : 0)) {
        // the rank-one coupling a e_last e_first^t, split as sqrt(a) on both sides so
        // that the two factors carry the same scale
        val = cvt<R>(csqrt(east[(long long)m * (g.n + 1) + edge]));
      }
      dst[(long long)col * s + i] = val;
    }
    if (blockIdx.y == 0 && threadIdx.x == 0) {
      S_rank[v] = k;
      G_rank[v] = 0;
    }
    return;
  }
  if (blockIdx.y > 0) return;
  __shared__ c128 A[8][16];
  __shared__ c128 colk[8];
  __shared__ int piv;
  __shared__ double s_red[4];
  const int lf = g.leaf, lam = nleaves + blockIdx.x, tid = threadIdx.x;
  const int lo = g.lo[lam], s = g.sz[lam];
  const bool act = tid < 128;         // four warps, one a scheduler (FP64)
  for (int e = tid; e < lf * 2 * lf; e += blockDim.x) {
    const int a = e / (2 * lf), b = e % (2 * lf);
    c128 v(0.0, 0.0);
    if (b >= lf) {
      v = c128(a == b - lf ? 1.0 : 0.0, 0.0);
    } else {
      Cx<R> x(0, 0);
      if (a < s && b < s) {
        const int i = lo + a, j = lo + b;
        c128 av(0, 0);
        if (a == b) av = diag[(long long)m * g.n + i];
        else if (j == i + 1) av = east[(long long)m * (g.n + 1) + j];
        else if (i == j + 1) av = east[(long long)m * (g.n + 1) + i];
        x = cvt<R>(av);
        if (Tprev) {
          const Cx<R> di = cvt<R>(north[(long long)m * g.n + i]), dj = cvt<R>(north[(long long)m * g.n + j]);
          x -= di * (Tprev[(long long)blockIdx.x * lf * lf + b * lf + a] * dj);
        }
      } else if (a == b) {
        x = Cx<R>(1, 0);    // identity padding keeps the padded leaf invertible
      }
      v = cvt<double>(x);
    }
    A[a][b] = v;
  }
  __syncthreads();
  // the largest squared modulus of the leaf's entries (one entry per thread, then warps)
  double scale2 = 0;
  if (act) {
    for (int e = tid; e < lf * lf; e += 128) scale2 = fmax(scale2, abs2(A[e / lf][e % lf]));
    for (int o = 16; o > 0; o >>= 1) scale2 = fmax(scale2, __shfl_xor_sync(0xffffffffu, scale2, o));
    if ((tid & 31) == 0) s_red[tid >> 5] = scale2;
  }
  __syncthreads();
  if (!act) return;
  // (from here on the first 128 threads, on their own barrier)
  auto sync = []() { asm volatile("bar.sync 1, 128;" ::: "memory"); };
  scale2 = fmax(fmax(s_red[0], s_red[1]), fmax(s_red[2], s_red[3]));
  bool bad = false;
  for (int k = 0; k < lf; ++k) {
    if (tid < 32) {
      // the first warp's lanes compare the candidates (ties: the smallest row)
      const int a = k + tid;
      double best = a < lf ? abs2(A[a][k]) : -1.0;
      int p = a < lf ? a : lf;
      for (int o = 4; o > 0; o >>= 1) {
        const double ob = __shfl_xor_sync(0xffffffffu, best, o);
        const int op = __shfl_xor_sync(0xffffffffu, p, o);
        if (ob > best || (ob == best && op < p)) { best = ob; p = op; }
      }
      if (tid == 0) piv = p;
    }
    sync();
    const int p = piv;
    if (p != k && tid < 2 * lf) {
      c128 t = A[k][tid]; A[k][tid] = A[p][tid]; A[p][tid] = t;
    }
    sync();
    const c128 pv = A[k][k];
    if (!(abs2(pv) > 1e-28 * scale2)) { bad = true; break; }   // |pivot| <= 1e-14 max |entry|
    const c128 ip = cinv_fast(pv);
    sync();
    if (tid < 2 * lf) A[k][tid] = A[k][tid] * ip;
    if (tid < lf) colk[tid] = A[tid][k];
    sync();
    for (int e = tid; e < lf * 2 * lf; e += 128) {
      const int a = e / (2 * lf), b = e % (2 * lf);
      if (a != k) A[a][b] = A[a][b] - colk[a] * A[k][b];
    }
    sync();
  }
  if (bad) {
    if (tid == 0) report_error(status, HSWEEP_ERR_NUMERIC, m);
    return;
  }
  Cx<R>* dst = G_leaf + (long long)blockIdx.x * lf * lf;
  for (int e = tid; e < lf * lf; e += 128) {
    const int a = e % lf, b = e / lf;
    dst[e] = cvt<R>(A[a][lf + b]);
  }
}

// ---------------------------------------------------------------------------------
// Y_v = G_v X_v for every node v at depth d+1 (X_v = S factor of v, k_v columns):
// an H-matrix times a tall-skinny block, as reductions (per node u below depth d+1:
// Qr_u = F_u^t X restricted to u) followed by an expansion.  Both are chains of dependent
// loads; they are cut short by spreading them over more CTAs and warps: the reductions take
// eight columns of X per CTA, the expansion 32 rows and four columns with the sum over the
// factor columns split over the eight warps (26.3 -> 8.9 us and 13.5 -> 6.4 us a
// launch at n = 511).
template <typename R>
__global__ void __launch_bounds__(kBlk) tsmm_reduce(Geo g, int d, const Cx<R>* __restrict__ G_F,
                                                    const int* __restrict__ G_rank, const Cx<R>* __restrict__ S_F,
                                                    const int* __restrict__ S_rank, Cx<R>* __restrict__ Qr) {
  pdl_begin();
  const int u = (1 << (d + 2)) + blockIdx.x;
  const int du = depth_of(u);
  const int nu = u >> (du - (d + 1));          // ancestor at depth d+1
  const int ru = G_rank[u], k = S_rank[nu], c0 = 8 * blockIdx.y;
  if (c0 >= k) return;
  const int s = g.sz[u], ld_x = g.sz[nu], xo = g.lo[u] - g.lo[nu];
  const Cx<R>* F = G_F + g.gfo[u];
  const Cx<R>* X[8];
#pragma unroll
  for (int t = 0; t < 8; ++t) X[t] = S_F + g.sfo[nu] + (long long)min(c0 + t, k - 1) * ld_x + xo;
  Cx<R>* out = Qr + g.qro[u];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  for (int kr = warp; kr < ru; kr += nw) {
    Cx<R> acc[8];
#pragma unroll
    for (int t = 0; t < 8; ++t) acc[t] = Cx<R>(0, 0);
    for (int i = lane; i < s; i += 32) {
      const Cx<R> f = F[(long long)kr * s + i];
#pragma unroll
      for (int t = 0; t < 8; ++t) cfma(acc[t], f, X[t][i]);
    }
    int t;
    bool first;
    scatter_sum<R, 8, 32, 1>(acc, lane, t, first);
    if (first && c0 + t < k) out[kr * g.KCAP + c0 + t] = acc[0];
  }
}

template <typename R>
__global__ void __launch_bounds__(kBlk) tsmm_expand(Geo g, int d, const Cx<R>* __restrict__ G_leaf,
                                                    const Cx<R>* __restrict__ G_F, const int* __restrict__ G_rank,
                                                    const Cx<R>* __restrict__ S_F, const int* __restrict__ S_rank,
                                                    const Cx<R>* __restrict__ Qr, Cx<R>* __restrict__ Y) {
  pdl_begin();
  __shared__ Cx<R> red[kBlk / 32][4][32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = kBlk / 32;
  const int row = min(blockIdx.x * 32 + lane, g.n - 1);
  const int col = 4 * blockIdx.y;
  const int lam = g.rowleaf[row];
  const int nu = lam >> (g.L - (d + 1));
  const int k = S_rank[nu];
  const int lo_nu = g.lo[nu], ld = g.sz[nu];
  Cx<R> y[4];
#pragma unroll
  for (int t = 0; t < 4; ++t) y[t] = Cx<R>(0, 0);
  if (col < k) {
    int ct[4];        // the columns (the last one again past the end)
#pragma unroll
    for (int t = 0; t < 4; ++t) ct[t] = min(col + t, k - 1);
    {
      const int lf = g.leaf, a = row - g.lo[lam], s = g.sz[lam];
      const Cx<R>* D = G_leaf + (long long)(lam - (1 << g.L)) * lf * lf;
      const Cx<R>* X = S_F + g.sfo[nu] + (g.lo[lam] - lo_nu);
      for (int b = warp; b < s; b += nw) {
        const Cx<R> f = D[b * lf + a];
#pragma unroll
        for (int t = 0; t < 4; ++t) cfma(y[t], f, X[(long long)ct[t] * ld + b]);
      }
    }
    for (int du = d + 2; du <= g.L; ++du) {
      const int u = lam >> (g.L - du);
      const int ru = G_rank[u];
      const Cx<R>* F = G_F + g.gfo[u] + (row - g.lo[u]);
      const Cx<R>* q = Qr + g.qro[u ^ 1];
      const int s = g.sz[u];
#pragma unroll 4
      for (int kr = warp; kr < ru; kr += nw) {
        const Cx<R> f = F[(long long)kr * s];
#pragma unroll
        for (int t = 0; t < 4; ++t) cfma(y[t], f, q[kr * g.KCAP + ct[t]]);
      }
    }
  }
#pragma unroll
  for (int t = 0; t < 4; ++t) red[warp][t][lane] = y[t];
  __syncthreads();
  const int t = threadIdx.x >> 5;       // column of this thread's sum
  if (t < 4 && blockIdx.x * 32 + lane < g.n && col + t < k) {
    Cx<R> v = red[0][t][lane];
#pragma unroll
    for (int w = 1; w < kBlk / 32; ++w) v += red[w][t][lane];
    Y[(long long)lo_nu * g.KCAP + (long long)(col + t) * ld + (row - lo_nu)] = v;
  }
}

// ---------------------------------------------------------------------------------
// Woodbury core per node t at depth d: P = U^t Y_a, Q = V^t Y_b (k x k), then
// M = [[P, I], [I, Q]]^{-1} by in-place Gauss-Jordan with partial pivoting.
template <typename R>
__global__ void core_dots(Geo g, int d, const Cx<R>* __restrict__ S_F, const int* __restrict__ S_rank,
                          const Cx<R>* __restrict__ Y, Cx<R>* __restrict__ PQ) {
  pdl_begin();
  const int t = (1 << d) + blockIdx.x / 2;
  const int side = blockIdx.x & 1;
  const int v = 2 * t + side;
  const int k = S_rank[v], s = g.sz[v];
  const Cx<R>* U = S_F + g.sfo[v];
  const Cx<R>* Yv = Y + (long long)g.lo[v] * g.KCAP;
  Cx<R>* out = PQ + ((long long)(t - (1 << d)) * 2 + side) * g.KCAP * g.KCAP;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  const int kb = (k + 3) / 4;      // four columns of Y at a time
  for (int e = blockIdx.y * nw + warp; e < k * kb; e += gridDim.y * nw) {
    const int a = e / kb, b = 4 * (e % kb);
    Cx<R> acc[4];
    const Cx<R>* yc[4];
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      acc[t] = Cx<R>(0, 0);
      yc[t] = Yv + (long long)min(b + t, k - 1) * s;
    }
    for (int i = lane; i < s; i += 32) {
      const Cx<R> f = U[(long long)a * s + i];
#pragma unroll
      for (int t = 0; t < 4; ++t) cfma(acc[t], f, yc[t][i]);
    }
    int t;
    bool first;
    scatter_sum<R, 4, 32, 1>(acc, lane, t, first);
    if (first && b + t < k) out[a * g.KCAP + b + t] = acc[0];
  }
}

// (the whole CTA; dynamic shared memory sm)
template <typename R>
__device__ void core_inverse_pivoted(const Geo& g, int d, int m, const int* __restrict__ S_rank,
                                     const Cx<R>* __restrict__ PQ, Cx<R>* __restrict__ Mb, int* status,
                                     unsigned char* sm) {
  const int t = (1 << d) + blockIdx.x;
  const int k = S_rank[2 * t];
  const int n2 = 2 * k;
  Cx<R>* A = reinterpret_cast<Cx<R>*>(sm);                 // n2 x n2, row-major
  R* red = reinterpret_cast<R*>(A + n2 * n2);              // [32]
  int* piv = reinterpret_cast<int*>(red + 32);             // [n2]
  __shared__ int s_p;
  __shared__ R s_best;
  const Cx<R>* P = PQ + ((long long)(t - (1 << d)) * 2) * g.KCAP * g.KCAP;
  const Cx<R>* Q = P + g.KCAP * g.KCAP;
  for (int e = threadIdx.x; e < n2 * n2; e += blockDim.x) {
    const int a = e / n2, b = e % n2;
    Cx<R> v(0, 0);
    if (a < k && b < k) v = P[a * g.KCAP + b];
    else if (a >= k && b >= k) v = Q[(a - k) * g.KCAP + (b - k)];
    else if (a < k && b == a + k) v = Cx<R>(1, 0);
    else if (a >= k && b == a - k) v = Cx<R>(1, 0);
    A[e] = v;
  }
  R mx = 0;
  for (int e = threadIdx.x; e < n2 * n2; e += blockDim.x) mx = fmax(mx, abs2(A[e]));
  __syncthreads();
  // block max
  {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    for (int o = 16; o > 0; o >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if (lane == 0) red[warp] = mx;
    __syncthreads();
    mx = 0;
    for (int i = 0; i < nw; ++i) mx = fmax(mx, red[i]);
    __syncthreads();
  }
  const R tiny = (sizeof(R) == 8 ? R(1e-30) : R(1e-14)) * mx;   // on |pivot|^2
  bool bad = false;
  // Gauss-Jordan in place, three block barriers per column: (1) pivot search and the
  // pivot's inverse, (2) the row interchange with the normalisation of the pivot row, (3)
  // the elimination of the other rows, each row owned by a group of gT lanes of one warp
  // (the group reads its multiplier, synchronises, then updates its columns, the pivot
  // column included)
  int gT = 1;
  while (gT < 32 && 2 * gT * n2 <= (int)blockDim.x) gT *= 2;
  const int rows_per_pass = (int)blockDim.x / gT;
  __shared__ Cx<R> s_ip;
  for (int kk = 0; kk < n2; ++kk) {
    if (threadIdx.x < 32) {
      // partial pivoting: warp 0 finds the largest |A[a][kk]|, a >= kk (ties: the smallest a)
      int p = n2;
      R best = R(-1);
      for (int a = kk + (int)threadIdx.x; a < n2; a += 32) {
        const R v = abs2(A[a * n2 + kk]);
        if (v > best) { best = v; p = a; }
      }
      for (int o = 16; o > 0; o >>= 1) {
        const R ob = __shfl_xor_sync(0xffffffffu, best, o);
        const int op = __shfl_xor_sync(0xffffffffu, p, o);
        if (ob > best || (ob == best && op < p)) { best = ob; p = op; }
      }
      if (threadIdx.x == 0) {
        s_p = p;
        s_best = best;
        piv[kk] = p;
        if (best > tiny) s_ip = cinv(A[p * n2 + kk]);
      }
    }
    __syncthreads();                                                     // (1)
    if (!(s_best > tiny)) { bad = true; break; }
    const int p = s_p;
    const Cx<R> ip = s_ip;
    for (int b = threadIdx.x; b < n2; b += blockDim.x) {
      const Cx<R> tk = A[kk * n2 + b], tp = A[p * n2 + b];
      if (p != kk) A[p * n2 + b] = tk;
      A[kk * n2 + b] = ((b == kk) ? Cx<R>(1, 0) : tp) * ip;
    }
    __syncthreads();                                                     // (2)
    for (int a0 = 0; a0 < n2; a0 += rows_per_pass) {
      const int a = a0 + (int)threadIdx.x / gT, sub = (int)threadIdx.x % gT;
      const bool live = a < n2 && a != kk;
      const Cx<R> f = live ? A[a * n2 + kk] : Cx<R>(0, 0);
      __syncwarp();
      if (live)
        for (int b = sub; b < n2; b += gT)
          A[a * n2 + b] = (b == kk) ? -(f * ip) : A[a * n2 + b] - f * A[kk * n2 + b];
    }
    __syncthreads();                                                     // (3)
  }
  if (bad) {
    if (threadIdx.x == 0) report_error(status, HSWEEP_ERR_NUMERIC, m);
    return;
  }
  // undo the row interchanges as column interchanges, in reverse order
  for (int kk = n2 - 1; kk >= 0; --kk) {
    const int p = piv[kk];
    if (p != kk)
      for (int a = threadIdx.x; a < n2; a += blockDim.x) {
        Cx<R> tmp = A[a * n2 + kk]; A[a * n2 + kk] = A[a * n2 + p]; A[a * n2 + p] = tmp;
      }
    __syncthreads();
  }
  Cx<R>* M = Mb + (long long)(t - (1 << d)) * 4 * g.KCAP * g.KCAP;
  for (int e = threadIdx.x; e < n2 * n2; e += blockDim.x) {
    const int a = e / n2, b = e % n2;
    M[a * 2 * g.KCAP + b] = A[e];
  }
}

template <typename R>
__global__ void core_inverse(Geo g, int d, int m, const int* __restrict__ S_rank, const Cx<R>* __restrict__ PQ,
                             Cx<R>* __restrict__ Mb, int* status) {
  pdl_begin();
  extern __shared__ __align__(16) unsigned char sm[];
  core_inverse_pivoted<R>(g, d, m, S_rank, PQ, Mb, status, sm);
}

// In complex64, the blocks of the inverse that are used, from one k x k inverse: with
// N = (I - Q P)^{-1},
//     M11 = -N Q,  M12 = N,  M22 = -P N   (M21 = M12^t is not needed),
// half the pivots and an eighth of the elimination of the 2k x 2k matrix (33.8 -> 21.7
// us a depth at n = 511).  It takes the identity blocks as pivots, which is as stable as pivoting
// while the entries of P and Q are of order one, as they are for a block's coupling seen
// through its own inverse; a matrix with an entry above kCoreLarge, or with a vanishing pivot,
// goes through the pivoted elimination above.
// N by Gauss-Jordan in registers: warp w of sixteen holds the rows w, w + 16, ..., a lane the
// columns lane, lane + 32.  No row is moved: a pivot row keeps its place (order kept in prow)
// and the interchanges are undone by where the result is written.  After its update each warp
// offers its best candidate for the next pivot and that row; after one barrier every warp
// picks the largest of the sixteen offers.
constexpr int kCoreWarps = 16, kCoreRows = 4, kCoreCols = 2;      // k <= 57 columns (r_max + 1)
constexpr float kCoreLarge = 4.0f;

// out[i][j] = add[i][j] + sgn (X Y)[i][j] for k x k matrices in shared memory (ld k), 2 x 2 tiles
template <typename Store>
__device__ __forceinline__ void core_gemm(const Cx<float>* X, const Cx<float>* Y, int k, Store store) {
  const int kt = (k + 1) / 2;
  for (int e = threadIdx.x; e < kt * kt; e += blockDim.x) {
    const int i0 = 2 * (e / kt), j0 = 2 * (e % kt), i1 = min(i0 + 1, k - 1), j1 = min(j0 + 1, k - 1);
    Cx<float> a00(0.f, 0.f), a01 = a00, a10 = a00, a11 = a00;
#pragma unroll 2
    for (int l = 0; l < k; ++l) {
      const Cx<float> x0 = X[i0 * k + l], x1 = X[i1 * k + l], y0 = Y[l * k + j0], y1 = Y[l * k + j1];
      cfma(a00, x0, y0);
      cfma(a01, x0, y1);
      cfma(a10, x1, y0);
      cfma(a11, x1, y1);
    }
    store(i0, j0, a00);
    if (j1 > j0) store(i0, j1, a01);
    if (i1 > i0) store(i1, j0, a10);
    if (i1 > i0 && j1 > j0) store(i1, j1, a11);
  }
}

__global__ void __launch_bounds__(32 * kCoreWarps) core_inverse_block(Geo g, int d, int m,
                                                                      const int* __restrict__ S_rank,
                                                                      const Cx<float>* __restrict__ PQ,
                                                                      Cx<float>* __restrict__ Mb, int* status) {
  pdl_begin();
  extern __shared__ __align__(16) unsigned char sm[];
  __shared__ Cx<float> offer[2][kCoreWarps][32 * kCoreCols];
  __shared__ float osize[2][kCoreWarps];
  __shared__ int orow[2][kCoreWarps];
  __shared__ int prow[kCoreWarps * kCoreRows];
  __shared__ float red[2][kCoreWarps];
  const int t = (1 << d) + blockIdx.x;
  const int k = S_rank[2 * t];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const Cx<float>* Pg = PQ + ((long long)(t - (1 << d)) * 2) * g.KCAP * g.KCAP;
  const Cx<float>* Qg = Pg + g.KCAP * g.KCAP;
  Cx<float>* P = reinterpret_cast<Cx<float>*>(sm);
  Cx<float>* Q = P + k * k;
  Cx<float>* B = Q + k * k;
  float mx = 0;
  for (int e = threadIdx.x; e < k * k; e += blockDim.x) {
    const int i = e / k, j = e - i * k;
    const Cx<float> p = Pg[i * g.KCAP + j], q = Qg[i * g.KCAP + j];
    P[e] = p;
    Q[e] = q;
    mx = fmaxf(mx, fmaxf(abs2(p), abs2(q)));
  }
  for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  if (lane == 0) red[0][warp] = mx;
  __syncthreads();
#pragma unroll
  for (int i = 0; i < kCoreWarps; ++i) mx = fmaxf(mx, red[0][i]);
  if (!(mx <= kCoreLarge * kCoreLarge)) {
    __syncthreads();
    core_inverse_pivoted<float>(g, d, m, S_rank, PQ, Mb, status, sm);
    return;
  }
  core_gemm(Q, P, k, [&](int i, int j, Cx<float> v) { B[i * k + j] = (i == j ? Cx<float>(1.f, 0.f) : Cx<float>(0.f, 0.f)) - v; });
  __syncthreads();
  Cx<float> A[kCoreRows][kCoreCols];
  mx = 0;
#pragma unroll
  for (int r = 0; r < kCoreRows; ++r)
#pragma unroll
    for (int c = 0; c < kCoreCols; ++c) {
      const int a = warp + kCoreWarps * r, b = lane + 32 * c;
      A[r][c] = (a < k && b < k) ? B[a * k + b] : Cx<float>(0.f, 0.f);
      mx = fmaxf(mx, abs2(A[r][c]));
    }
  for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  if (lane == 0) red[1][warp] = mx;
  const int nr = (k - warp + kCoreWarps - 1) / kCoreWarps;      // rows of this warp
  unsigned used = 0;                    // bit r: row r of this warp was a pivot row
  // this warp's largest unused |A[.][kl + 32 cc]|^2 (ties: the smallest row) and that row
  auto make_offer = [&](auto ccc, int kl, int b) {
    constexpr int cc = decltype(ccc)::value;
    float best = -1.f;
    int br = 0;
#pragma unroll
    for (int r = 0; r < kCoreRows; ++r) {
      const float v = abs2(A[r][cc]);
      if (r < nr && !(used >> r & 1u) && v > best) { best = v; br = r; }
    }
    best = __shfl_sync(0xffffffffu, best, kl);      // the lane that holds the column decides
    br = __shfl_sync(0xffffffffu, br, kl);
    if (lane == 0) {
      osize[b][warp] = best;
      orow[b][warp] = warp + kCoreWarps * br;
    }
#pragma unroll
    for (int r = 0; r < kCoreRows; ++r)
      if (r == br) {
#pragma unroll
        for (int c = 0; c < kCoreCols; ++c) offer[b][warp][lane + 32 * c] = A[r][c];
      }
  };
  make_offer(std::integral_constant<int, 0>(), 0, 0);
  __syncthreads();
  mx = 0;
#pragma unroll
  for (int i = 0; i < kCoreWarps; ++i) mx = fmaxf(mx, red[1][i]);
  const float tiny = 1e-14f * mx;       // on |pivot|^2
  bool bad = false;
  auto half = [&](auto ccc) {           // the pivots of columns 32 cc ..
    constexpr int cc = decltype(ccc)::value;
    for (int kk = 32 * cc; kk < min(k, 32 * cc + 32); ++kk) {
      const int b = kk & 1, kl = kk & 31;
      float best = osize[b][0];
      int ow = 0, p = orow[b][0];
#pragma unroll
      for (int i = 1; i < kCoreWarps; ++i) {
        const float v = osize[b][i];
        const int pi = orow[b][i];
        if (v > best || (v == best && pi < p)) { best = v; ow = i; p = pi; }
      }
      if (!(best > tiny)) { bad = true; return; }
      if (threadIdx.x == 0) prow[kk] = p;
      const Cx<float> ip = cinv(offer[b][ow][kk]);
      // the pivot row divided by the pivot, with 1 / pivot in its own column
      Cx<float> pr[kCoreCols];
#pragma unroll
      for (int c = 0; c < kCoreCols; ++c) pr[c] = offer[b][ow][lane + 32 * c] * ip;
      if (lane == kl) pr[cc] = ip;
#pragma unroll
      for (int r = 0; r < kCoreRows; ++r) {
        if (r < nr) {
          const Cx<float> f(__shfl_sync(0xffffffffu, A[r][cc].re, kl), __shfl_sync(0xffffffffu, A[r][cc].im, kl));
          if (warp + kCoreWarps * r == p) {
            used |= 1u << r;
#pragma unroll
            for (int c = 0; c < kCoreCols; ++c) A[r][c] = pr[c];
          } else {
            if (lane == kl) A[r][cc] = Cx<float>(0.f, 0.f);
#pragma unroll
            for (int c = 0; c < kCoreCols; ++c) cfma(A[r][c], -f, pr[c]);
          }
        }
      }
      if (kk + 1 < k) {
        if (kl < 31) make_offer(ccc, kl + 1, b ^ 1);
        else make_offer(std::integral_constant<int, (cc + 1 < kCoreCols ? cc + 1 : cc)>(), 0, b ^ 1);
      }
      __syncthreads();
    }
  };
  half(std::integral_constant<int, 0>());
  if (!bad && k > 32) half(std::integral_constant<int, 1>());
  if (bad) {
    __syncthreads();
    core_inverse_pivoted<float>(g, d, m, S_rank, PQ, Mb, status, sm);
    return;
  }
  // physical row prow[i] is row i of the inverse, column l is its column prow[l]
  int* inv = reinterpret_cast<int*>(&offer[0][0][0]);      // logical row of a physical one
  for (int i = threadIdx.x; i < k; i += blockDim.x) inv[prow[i]] = i;
  __syncthreads();
  Cx<float>* M = Mb + (long long)(t - (1 << d)) * 4 * g.KCAP * g.KCAP;
  const int ldm = 2 * g.KCAP;
#pragma unroll
  for (int r = 0; r < kCoreRows; ++r)
    if (r < nr) {
      const int i = inv[warp + kCoreWarps * r];
#pragma unroll
      for (int c = 0; c < kCoreCols; ++c) {
        const int l = lane + 32 * c;
        if (l < k) {
          B[i * k + prow[l]] = A[r][c];
          M[i * ldm + k + prow[l]] = A[r][c];                  // M12
        }
      }
    }
  __syncthreads();
  core_gemm(B, Q, k, [&](int i, int j, Cx<float> v) { M[i * ldm + j] = -v; });                       // M11
  core_gemm(P, B, k, [&](int i, int j, Cx<float> v) { M[(k + i) * ldm + k + j] = -v; });             // M22
}

// W_v = Y_v M_side (k x k block of M), and the new off-diagonal block at the parent:
// F_a = -Y_a M12, F_b = Y_b.  A thread has one entry of each; what bounds it is the latency of
// its chain of loads, so eight terms are loaded at a time (6.7 us a launch at n = 511; with four
// columns a thread, which read Y a quarter as often, 11.3).
template <typename R>
__global__ void __launch_bounds__(128) woodbury_form(Geo g, int d, const int* __restrict__ S_rank,
                                                     const Cx<R>* __restrict__ Y, const Cx<R>* __restrict__ Mb,
                                                     Cx<R>* __restrict__ W, Cx<R>* __restrict__ G_F,
                                                     int* __restrict__ G_rank) {
  pdl_begin();
  const int row = blockIdx.x * 32 + (threadIdx.x & 31);
  const int col = blockIdx.y * 4 + (threadIdx.x >> 5);
  if (row >= g.n) return;
  const int v = g.rowleaf[row] >> (g.L - (d + 1));
  const int t = v >> 1, side = v & 1;
  const int k = S_rank[v];
  if (col >= k) return;
  const int s = g.sz[v], i = row - g.lo[v];
  const Cx<R>* Yv = Y + (long long)g.lo[v] * g.KCAP + i;
  const int ldm = 2 * g.KCAP;
  const Cx<R>* M2 = Mb + (long long)(t - (1 << d)) * 4 * g.KCAP * g.KCAP + k + col;     // M12
  const Cx<R>* M1 = M2 + (side ? k * ldm : -k);                                        // M22 or M11
  Cx<R> w(0, 0), nf(0, 0);
#pragma unroll 8
  for (int j = 0; j < k; ++j) {
    const Cx<R> y = Yv[(long long)j * s];
    cfma(w, y, M1[j * ldm]);
    if (!side) cfma(nf, y, M2[j * ldm]);
  }
  W[(long long)g.lo[v] * g.KCAP + (long long)col * s + i] = w;
  G_F[g.gfo[v] + (long long)col * s + i] = side ? Yv[(long long)col * s] : -nf;
  if (i == 0 && col == 0) G_rank[v] = k;
}

// Append the rank-k correction to every node below depth d+1 and update the leaves
// (a leaf at depth d+1 itself only gets the dense update; its factor slot holds the
// new block written by woodbury_form).
template <typename R>
__global__ void woodbury_append(Geo g, int d, const int* __restrict__ S_rank, const Cx<R>* __restrict__ Y,
                                const Cx<R>* __restrict__ W, Cx<R>* __restrict__ G_F, int* __restrict__ G_rank,
                                Cx<R>* __restrict__ G_leaf) {
  pdl_begin();
  const int u = (1 << (d + 1)) + blockIdx.x;
  const int du = depth_of(u);
  const int nu = u >> (du - (d + 1));
  const int k = S_rank[nu];
  const bool append = du >= d + 2;
  const int r0 = append ? G_rank[u] : 0;
  const int s = g.sz[u], ld = g.sz[nu], xo = g.lo[u] - g.lo[nu];
  const Cx<R>* Yv = Y + (long long)g.lo[nu] * g.KCAP;
  const Cx<R>* Wv = W + (long long)g.lo[nu] * g.KCAP;
  const bool left = (u & 1) == 0;
  Cx<R>* F = G_F + g.gfo[u];
  if (append)
    for (int e = threadIdx.x; e < s * k; e += blockDim.x) {
      const int i = e % s, j = e / s;
      F[(long long)(r0 + j) * s + i] = left ? -Wv[(long long)j * ld + xo + i] : Yv[(long long)j * ld + xo + i];
    }
  if (du == g.L) {     // leaf: G_leaf -= W[leaf] Y[leaf]^t
    const int lf = g.leaf;
    Cx<R>* D = G_leaf + (long long)(u - (1 << g.L)) * lf * lf;
    for (int e = threadIdx.x; e < s * s; e += blockDim.x) {
      const int a = e % s, b = e / s;
      Cx<R> acc(0, 0);
      for (int j = 0; j < k; ++j) cfma(acc, Wv[(long long)j * ld + xo + a], Yv[(long long)j * ld + xo + b]);
      D[b * lf + a] -= acc;
    }
  }
  __syncthreads();
  if (append && threadIdx.x == 0) G_rank[u] = r0 + k;
}

// ---------------------------------------------------------------------------------
// lanes per column of the Gram-Schmidt steps
template <typename R> __host__ __device__ constexpr int group_lanes() { return sizeof(R) == 8 ? 8 : 32; }

// Recompression, step 1, for the nodes u = list[blockIdx.x]: with w = rank(u) columns,
// a factor with at least as many columns as rows (w >= sz(u)), or in complex64 of at most
// kDenseRows rows, takes the dense path, Q = I and R = F_u (qcols = sz(u), qmode = 1);
// otherwise the QR of F_u in place by modified Gram-Schmidt: a column whose remainder is at
// the rounding level of its own norm is dropped, the Q columns are compacted and R (qc x w)
// written out (qmode = 0).  R is row-major with leading dimension cap(u).
// Every step updates all later columns (a warp per column, the new norm with the update), so
// a step costs one barrier; classical Gram-Schmidt with its two passes took ten, 3.6 us a
// column (the launch at n = 511: 316 us, now 54; n = 150 in complex128: 931, now 360).  A column
// of which less than kReorth is left when its turn comes is orthogonalised once more against all
// Q columns before it (two barriers).  Without that the skews compound: each column takes over
// those of the columns subtracted from it, enlarged by what it lost, and cosines of 0.05 to 0.8
// were reached on columns with remainders of a tenth each.  F = Q R holds to rounding either way;
// the singular values of the core are those of the block only as far as Q is orthogonal.  When F_u
// fits the kernel's shared memory (qs_entries) the columns stay there.
constexpr float kReorth = 0.5f;
// bytes of the tables in front of the columns
template <typename R> __host__ __device__ constexpr size_t qr_tables(int wcap) {
  return ((size_t)wcap * (3 * sizeof(R) + sizeof(Cx<R>) + sizeof(int)) + 15) & ~size_t(15);
}
template <typename R>
__global__ void __launch_bounds__(1024) qr_mgs(Geo g, Cx<R>* __restrict__ G_F, const int* __restrict__ G_rank,
                                               Cx<R>* __restrict__ Rb, int* __restrict__ qcols, int* __restrict__ qmode,
                                               int qs_entries) {
  pdl_begin();
  extern __shared__ __align__(16) unsigned char sm[];
  const int u = g.list[blockIdx.x];
  const int s = g.sz[u], w = G_rank[u], ld = g.cap[u];
  Cx<R>* F = G_F + g.gfo[u];
  Cx<R>* Rm = Rb + g.rbo[u];                               // row-major qc x w, ld cap(u)
  if (s <= g.QCAP && (w >= s || s <= g.dense_max)) {
    for (int e = threadIdx.x; e < s * w; e += blockDim.x) {
      const int i = e % s, l = e / s;
      Rm[(long long)i * ld + l] = F[e];
    }
    if (threadIdx.x == 0) { qcols[u] = s; qmode[u] = 1; }
    return;
  }
  const int wcap = g.cap_max;
  Cx<R>* co = reinterpret_cast<Cx<R>*>(sm);                // [wcap] coefficients of a second pass
  R* cur = reinterpret_cast<R*>(co + wcap);                // [wcap] squared norm of a column's remainder
  R* org = cur + wcap;                                     // [wcap] and of the column itself
  R* rn = org + wcap;                                      // [wcap] 1 / norm of a Q column's source
  int* src = reinterpret_cast<int*>(rn + wcap);            // [wcap] and that source
  __shared__ R red[32];
  const bool qsh = (long long)s * w <= qs_entries;
  Cx<R>* Fq = qsh ? reinterpret_cast<Cx<R>*>(sm + qr_tables<R>(wcap)) : F;   // the columns being orthogonalised
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  const int rows = min(s, ld);
  for (int e = threadIdx.x; e < rows * w; e += blockDim.x) Rm[(long long)(e / w) * ld + e % w] = Cx<R>(0, 0);
  for (int j = warp; j < w; j += nw) {
    R acc = 0;
    for (int i = lane; i < s; i += 32) {
      const Cx<R> v = F[(long long)j * s + i];
      if (qsh) Fq[(long long)j * s + i] = v;
      acc += abs2(v);
    }
    acc = warp_sum_r(acc);
    if (lane == 0) cur[j] = org[j] = acc;
  }
  __syncthreads();
  constexpr int kGL = group_lanes<R>(), kCPW = 32 / kGL;
  int qc = 0;
  for (int j = 0; j < w; ++j) {
    R nr = cur[j];
    bool kept = nr > Tiny<R>::dep * Tiny<R>::dep * org[j] && nr > 0 && qc < rows;
    if (kept && qc > 0 && nr < R(kReorth * kReorth) * org[j]) {
      Cx<R>* cj = Fq + (long long)j * s;
      for (int kb = warp * kCPW; kb < qc; kb += nw * kCPW) {
        const int k = kb + lane / kGL, gl = lane % kGL;
        const bool act = k < qc;
        const Cx<R>* ck = Fq + (long long)src[act ? k : 0] * s;
        Cx<R> d(0, 0);
        if (act)
          for (int i = gl; i < s; i += kGL) cfma_conj(d, ck[i], cj[i]);
        for (int o = kGL / 2; o > 0; o >>= 1) d += shfl_xor(d, o);
        if (act && gl == 0) {
          d = rn[k] * d;
          co[k] = -(rn[k] * d);
          Rm[(long long)k * ld + j] += d;
        }
      }
      __syncthreads();
      // kRW neighbouring rows a warp (their words are in different banks whatever the column's
      // place), the columns over 32 / kRW groups of lanes
      constexpr int kRW = sizeof(R) == 8 ? 8 : 16;
      R part = 0;
      for (int i0 = kRW * warp; i0 < s; i0 += kRW * nw) {
        const int i = i0 + lane % kRW;
        Cx<R> v(0, 0);
        if (i < s) {
#pragma unroll 4
          for (int k = lane / kRW; k < qc; k += 32 / kRW) cfma(v, co[k], Fq[(long long)src[k] * s + i]);
        }
        for (int o = kRW; o < 32; o <<= 1) v += shfl_xor(v, o);
        if (i < s && lane < kRW) {
          v += cj[i];
          cj[i] = v;
          part += abs2(v);
        }
      }
      for (int o = 1; o < kRW; o <<= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
      if (lane == 0) red[warp] = part;
      __syncthreads();
      nr = warp_sum_r(lane < nw ? red[lane] : R(0));
      kept = nr > Tiny<R>::dep * Tiny<R>::dep * org[j] && nr > 0;
    }
    if (kept) {
      const R inv = rcp_any(nr), rs = rsqrt_any(nr), nn = nr * rs;
      const Cx<R>* cj = Fq + (long long)j * s;
      for (int lb = j + 1 + warp * kCPW; lb < w; lb += nw * kCPW) {
        const int l = lb + lane / kGL, gl = lane % kGL;
        const bool act = l < w;
        Cx<R>* cl = Fq + (long long)(act ? l : j) * s;
        Cx<R> d(0, 0);
        if (act)
          for (int i = gl; i < s; i += kGL) cfma_conj(d, cj[i], cl[i]);
        for (int o = kGL / 2; o > 0; o >>= 1) d += shfl_xor(d, o);
        const Cx<R> be = -(inv * d);
        R acc = 0;
        if (act)
          for (int i = gl; i < s; i += kGL) {
            Cx<R> v = cl[i];
            cfma(v, be, cj[i]);
            cl[i] = v;
            acc = fma(v.re, v.re, fma(v.im, v.im, acc));
          }
        for (int o = kGL / 2; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
        if (act && gl == 0) {
          cur[l] = acc;
          Rm[(long long)qc * ld + l] = rs * d;
        }
      }
      if (threadIdx.x == 0) {
        Rm[(long long)qc * ld + j] = Cx<R>(nn, 0);
        src[qc] = j;
        rn[qc] = rs;
      }
      ++qc;
    }
    __syncthreads();
  }
  // the kept columns, normalised, to the front (a Q column never lies behind its source)
  for (int c = 0; c < qc; ++c) {
    const int j = src[c];
    const R rs = rn[c];
    for (int i = threadIdx.x; i < s; i += blockDim.x) F[(long long)c * s + i] = rs * Fq[(long long)j * s + i];
    if (!qsh) __syncthreads();
  }
  if (threadIdx.x == 0) { qcols[u] = qc; qmode[u] = 0; }
}

// Recompression, step 2a: the cores C = R_a R_b^t (qa x qb, column-major, ld qa, at
// Cb + (a / 2) QCAP^2) of the sibling pairs a = list[blockIdx.y], one kCT x kCT tile of C
// per CTA (blockIdx.x).  Two kernels compute them: core_product_cc on CUDA cores (either
// precision) and, in complex64, core_product_tc on tensor cores; the setup times both on
// a layer of representative ranks and keeps the faster for each kind of recompression
// launch (factor_impl).
// tile edge in complex entries; in complex128 a quarter of the tile per CTA (FP64 units)
template <typename R> __host__ __device__ constexpr int core_tile_edge() { return sizeof(R) == 8 ? 16 : 32; }
constexpr int kCK = 16;    // complex k chunk staged in shared memory

template <int kCT>
__device__ __forceinline__ bool core_tile(int qa, int qb, int tile, int& ti, int& tj) {
  const int ni = (qa + kCT - 1) / kCT, nj = (qb + kCT - 1) / kCT;
  if (tile >= ni * nj) return false;
  ti = tile % ni;
  tj = tile / ni;
  return true;
}

// 256 threads: thread (tx, ty) of a 16 x 16 grid owns rows ty (+ 16) and columns tx (+ 16)
// of the tile; the k chunks of R_a and R_b are staged with coalesced loads
template <typename R>
__global__ void __launch_bounds__(256) core_product_cc(Geo g, const Cx<R>* __restrict__ Rb,
                                                       const int* __restrict__ qcols, const int* __restrict__ G_rank,
                                                       Cx<R>* __restrict__ Cb) {
  pdl_begin();
  constexpr int kCT = core_tile_edge<R>(), U = kCT / 16;
  __shared__ Cx<R> As[kCK][kCT + 1], Bs[kCK][kCT + 1];
  const int a = g.list[blockIdx.y], b = a + 1;
  const int qa = qcols[a], qb = qcols[b], w = G_rank[a];
  int ti, tj;
  if (!core_tile<kCT>(qa, qb, blockIdx.x, ti, tj)) return;
  const Cx<R>* Ra = Rb + g.rbo[a];
  const Cx<R>* Rbb = Rb + g.rbo[b];
  const int lda = g.cap[a], ldb = g.cap[b];
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  Cx<R> acc[U][U];
  for (int u = 0; u < U; ++u)
    for (int v = 0; v < U; ++v) acc[u][v] = Cx<R>(0, 0);
  for (int k0 = 0; k0 < w; k0 += kCK) {
    for (int e = threadIdx.x; e < kCK * kCT; e += blockDim.x) {
      const int kk = e % kCK, r = e / kCK;
      const int i = ti * kCT + r, j = tj * kCT + r, k = k0 + kk;
      As[kk][r] = (i < qa && k < w) ? Ra[(long long)i * lda + k] : Cx<R>(0, 0);
      Bs[kk][r] = (j < qb && k < w) ? Rbb[(long long)j * ldb + k] : Cx<R>(0, 0);
    }
    __syncthreads();
#pragma unroll 4
    for (int kk = 0; kk < kCK; ++kk)
#pragma unroll
      for (int u = 0; u < U; ++u)
#pragma unroll
        for (int v = 0; v < U; ++v) cfma(acc[u][v], As[kk][ty + 16 * u], Bs[kk][tx + 16 * v]);
    __syncthreads();
  }
  Cx<R>* C = Cb + (long long)(a >> 1) * g.QCAP * g.QCAP;
  for (int u = 0; u < U; ++u)
    for (int v = 0; v < U; ++v) {
      const int i = ti * kCT + ty + 16 * u, j = tj * kCT + tx + 16 * v;
      if (i < qa && j < qb) C[(long long)j * qa + i] = acc[u][v];
    }
}

// x = hi + lo with hi the TF32 rounding of x (10 explicit mantissa bits) and lo = x - hi,
// exact in FP32; a product in three TF32 parts, hi*hi + hi*lo + lo*hi with FP32
// accumulation, keeps about 2^-21 relative accuracy
__device__ __forceinline__ void tf32_split(float x, unsigned& hi, unsigned& lo) {
  hi = (__float_as_uint(x) + 0x1000u) & 0xffffe000u;
  lo = __float_as_uint(x - __uint_as_float(hi));
}
__device__ __forceinline__ void mma_m16n8k8_tf32(float (&c)[4], const unsigned (&a)[4], unsigned b0, unsigned b1) {
  asm volatile("mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
               : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
               : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// The complex product as one real product C' = A' B'^t: A' row i = (Re, Im) of row i of
// R_a interleaved (real k' = 2 l + q), and B' holds for output column n' = 2 j + p
//   B'[2l][2j] = Re b, B'[2l+1][2j] = -Im b, B'[2l][2j+1] = Im b, B'[2l+1][2j+1] = Re b
// (b = R_b[j][l]), so that C'[i][2j] = Re C[i][j] and C'[i][2j+1] = Im C[i][j].  Eight
// warps: warp (wm = warp & 1, wn = warp >> 1) owns tile rows 16 wm .. 16 wm + 15 and the
// real columns 16 wn .. 16 wn + 15 (two m16n8k8 column tiles).
__global__ void __launch_bounds__(256) core_product_tc(Geo g, const Cx<float>* __restrict__ Rb,
                                                       const int* __restrict__ qcols, const int* __restrict__ G_rank,
                                                       Cx<float>* __restrict__ Cb) {
  pdl_begin();
  constexpr int kCT = core_tile_edge<float>();
  __shared__ Cx<float> As[kCT][kCK + 1], Bs[kCT][kCK + 1];
  const int a = g.list[blockIdx.y], b = a + 1;
  const int qa = qcols[a], qb = qcols[b], w = G_rank[a];
  int ti, tj;
  if (!core_tile<kCT>(qa, qb, blockIdx.x, ti, tj)) return;
  const Cx<float>* Ra = Rb + g.rbo[a];
  const Cx<float>* Rbb = Rb + g.rbo[b];
  const int lda = g.cap[a], ldb = g.cap[b];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int wm = warp & 1, wn = warp >> 1;
  const int gid = lane >> 2, tig = lane & 3;
  float c[2][4] = {}, c2[2][4] = {};
  for (int k0 = 0; k0 < w; k0 += kCK) {
    for (int e = threadIdx.x; e < kCK * kCT; e += blockDim.x) {
      const int kk = e % kCK, r = e / kCK;
      const int i = ti * kCT + r, j = tj * kCT + r, k = k0 + kk;
      As[r][kk] = (i < qa && k < w) ? Ra[(long long)i * lda + k] : Cx<float>(0.f, 0.f);
      Bs[r][kk] = (j < qb && k < w) ? Rbb[(long long)j * ldb + k] : Cx<float>(0.f, 0.f);
    }
    __syncthreads();
    // real k' in steps of 8 over the chunk's 2 kCK real columns
#pragma unroll
    for (int ks = 0; ks < 2 * kCK; ks += 8) {
      // A fragment: rows 16 wm + gid (+ 8), real columns ks + tig (+ 4)
      unsigned ah[4], al[4];
      {
        const int r0 = 16 * wm + gid, r1 = r0 + 8;
        const int k1 = ks + tig, k2 = ks + tig + 4;
        const float v0 = (k1 & 1) ? As[r0][k1 >> 1].im : As[r0][k1 >> 1].re;
        const float v1 = (k1 & 1) ? As[r1][k1 >> 1].im : As[r1][k1 >> 1].re;
        const float v2 = (k2 & 1) ? As[r0][k2 >> 1].im : As[r0][k2 >> 1].re;
        const float v3 = (k2 & 1) ? As[r1][k2 >> 1].im : As[r1][k2 >> 1].re;
        tf32_split(v0, ah[0], al[0]);
        tf32_split(v1, ah[1], al[1]);
        tf32_split(v2, ah[2], al[2]);
        tf32_split(v3, ah[3], al[3]);
      }
#pragma unroll
      for (int nt = 0; nt < 2; ++nt) {
        // B fragment: real rows ks + tig (+ 4), real output column 16 wn + 8 nt + gid
        const int np = 16 * wn + 8 * nt + gid;
        const int j = np >> 1, p = np & 1;
        float bv[2];
#pragma unroll
        for (int h2 = 0; h2 < 2; ++h2) {
          const int kp = ks + tig + 4 * h2;
          const Cx<float> bb = Bs[j][kp >> 1];
          const int q = kp & 1;
          bv[h2] = p == 0 ? (q == 0 ? bb.re : -bb.im) : (q == 0 ? bb.im : bb.re);
        }
        unsigned bh0, bl0, bh1, bl1;
        tf32_split(bv[0], bh0, bl0);
        tf32_split(bv[1], bh1, bl1);
        mma_m16n8k8_tf32(c[nt], ah, bh0, bh1);
        mma_m16n8k8_tf32(c2[nt], al, bh0, bh1);
        mma_m16n8k8_tf32(c2[nt], ah, bl0, bl1);
      }
    }
    __syncthreads();
  }
  Cx<float>* C = Cb + (long long)(a >> 1) * g.QCAP * g.QCAP;
#pragma unroll
  for (int nt = 0; nt < 2; ++nt) {
    const int j = tj * kCT + ((16 * wn + 8 * nt) >> 1) + tig;   // output columns 2 tig, 2 tig + 1 of the n-tile
    const int i0 = ti * kCT + 16 * wm + gid, i1 = i0 + 8;
    if (j < qb) {
      if (i0 < qa) C[(long long)j * qa + i0] = Cx<float>(c[nt][0] + c2[nt][0], c[nt][1] + c2[nt][1]);
      if (i1 < qa) C[(long long)j * qa + i1] = Cx<float>(c[nt][2] + c2[nt][2], c[nt][3] + c2[nt][3]);
    }
  }
}

// Shuffle-sum within aligned groups of GW lanes (GW = 16 or 32).
template <typename R> __device__ __forceinline__ Cx<R> group_sum(Cx<R> v, int GW) {
  for (int o = GW >> 1; o > 0; o >>= 1) v += shfl_xor(v, o);
  return v;
}

// A bound on the squared spectral norm of the columns of C with nr >= 0 (squared norms nr): the
// Frobenius norm of their Gram matrix.  It is the Frobenius bound for aligned columns, and a sixth of
// it for 70 unrelated ones.  Whole CTA; a warp takes a column against four later ones at a time (10 us
// for 100 columns of 128).
__device__ __noinline__ float left_norm2(const Cx<float>* C, int ld, int qa, int qb, const float* nr, float* red) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  float sum = 0;
  for (int i = warp; i < qb; i += nw) {
    if (nr[i] < 0) continue;
    const Cx<float>* ci = C + i * ld;
    if (lane == 0) sum += nr[i] * nr[i];
    for (int j0 = i + 1; j0 < qb; j0 += 4) {
      Cx<float> d[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) d[u] = Cx<float>(0.f, 0.f);
      for (int r = lane; r < qa; r += 32) {
        const Cx<float> x = ci[r];
#pragma unroll
        for (int u = 0; u < 4; ++u) cfma_conj(d[u], x, C[min(j0 + u, qb - 1) * ld + r]);
      }
      int u;
      bool first;
      scatter_sum<float, 4, 32, 1>(d, lane, u, first);
      if (first && j0 + u < qb && nr[j0 + u] >= 0) sum += 2.0f * abs2(d[0]);
    }
  }
  sum = warp_sum_r(sum);
  if (lane == 0) red[warp] = sum;
  __syncthreads();
  sum = warp_sum_r(lane < nw ? red[lane] : 0.f);
  __syncthreads();
  return sqrtf(sum);
}

// Recompression, step 2b: for every sibling pair (a, b) with a = list[blockIdx.x], the
// truncated SVD of the core C (step 2a), as the small transforms
//   T_b = conj(P) Sigma^(1/2) (qb x k'),  T_a = C P Sigma^(-1/2) (qa x k'),
// P the right singular vectors kept: T_a T_b^t = C P P^*, the projection of C.
//
// 1. Gram-Schmidt with column pivoting, C = Q R, stopped when the squared norms of the
//    remaining columns sum to at most rem (relative to the largest column's), or to the rounding
//    noise of the core, or (complex64) when their Gram matrix shows that they are many unrelated
//    small ones: no singular value above sqrt(rem) is left behind, however the remaining columns
//    are aligned.  The block's numerical rank is a third to a half of the core's size.
//    Each warp picks the pivot from the column norms (no
//    broadcast), takes its columns' inner products with the pivot column, updates them and
//    leaves their new norms: one barrier a step.  Q is not kept: row k of R, conjugated, goes
//    into the storage of the k-th pivot column.
// 2. One-sided Jacobi on L = R^* (qb x kq): L W = P Sigma.  The rows of R come graded, so few
//    sweeps do.  No rotations are accumulated: T_a takes the product with C instead, and as
//    a projection of C it does not depend on how exactly the rotations were unitary (their
//    angles come from FP32 reciprocal square roots in both precisions).
// What bounds it is the latency of kq - 1 barriers a sweep (complex64) or the FP64 units of
// one SM (complex128).  A launch takes 205 us at n = 511 in complex64 (595 with Jacobi on
// the whole core, rotations accumulated), 324 us at n = 150 in complex128 (1612).
template <typename R>
__global__ void __launch_bounds__(1024) svd_jacobi(Geo g, double eps, const Cx<R>* __restrict__ Cb,
                                                   const int* __restrict__ qcols, Cx<R>* __restrict__ Tx,
                                                   int* __restrict__ newrank, int smem_entries, R thr, float rem) {
  pdl_begin();
  extern __shared__ __align__(16) unsigned char sm[];
  const int a = g.list[blockIdx.x], b = a + 1, t = a >> 1;
  const int qa = qcols[a], qb = qcols[b];
  const int ld = max(qa, qb);
  Cx<R>* C = reinterpret_cast<Cx<R>*>(sm);                        // column j at j ld
  Cx<R>* rbuf = C + smem_entries;                                  // [2][QCAP] a row of R
  R* nrm = reinterpret_cast<R*>(rbuf + 2 * g.QCAP);                // [2][QCAP] squared column norms
  R* sig = nrm + 2 * g.QCAP;                                       // [QCAP + 1]
  int* slot = reinterpret_cast<int*>(sig + g.QCAP + 1);            // [QCAP] column storage of row k
  int* order = slot + g.QCAP;                                      // [QCAP]
  __shared__ int s_rot, s_gg, s_t, s_keep;
  __shared__ float red[32];
  if (qa == 0 || qb == 0) {
    if (threadIdx.x == 0) { newrank[a] = 0; newrank[b] = 0; }
    return;
  }
  const Cx<R>* Cg = Cb + (long long)t * g.QCAP * g.QCAP;           // the core from step 2a
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  for (int j = warp; j < qb; j += nw) {
    R acc = 0;
    for (int i = lane; i < qa; i += 32) {
      const Cx<R> v = Cg[(long long)j * qa + i];
      C[j * ld + i] = v;
      acc += abs2(v);
    }
    acc = warp_sum_r(acc);
    if (lane == 0) nrm[j] = acc;
  }
  __syncthreads();
  // normalise by the largest column norm
  R mx = 0, tot = 0;
  for (int j = lane; j < qb; j += 32) {
    mx = fmax(mx, nrm[j]);
    tot += nrm[j];
  }
  for (int o = 16; o > 0; o >>= 1) {
    mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    tot += __shfl_xor_sync(0xffffffffu, tot, o);
  }
  if (!(mx > 0)) {
    if (threadIdx.x == 0) { newrank[a] = 0; newrank[b] = 0; }
    return;
  }
  const R scale = sqrt(mx), iscale = R(1) / scale;
  rem = fmaxf(rem, (float)(R(Tiny<R>::neg) * (tot / mx)));
  __syncthreads();
  for (int j = warp; j < qb; j += nw) {
    for (int i = lane; i < qa; i += 32) C[j * ld + i] = iscale * C[j * ld + i];
    if (lane == 0) nrm[j] = iscale * iscale * nrm[j];
  }
  __syncthreads();
  constexpr int kGL = group_lanes<R>(), kCPW = 32 / kGL;
  // ---- 1. pivoted Gram-Schmidt -----------------------------------------------------------
  int kq = 0;
  float check = FLT_MAX;
  const int kmax = min(qa, qb);
  for (; kq < kmax; ++kq) {
    const R* nr = nrm + (kq & 1) * g.QCAP;
    R* nx = nrm + ((kq & 1) ^ 1) * g.QCAP;
    Cx<R>* rk = rbuf + (kq & 1) * g.QCAP;
    R best = R(-1);
    int p = 0;
    for (int j = lane; j < qb; j += 32)
      if (nr[j] > best) { best = nr[j]; p = j; }
    for (int o = 16; o > 0; o >>= 1) {
      const R ob = __shfl_xor_sync(0xffffffffu, best, o);
      const int op = __shfl_xor_sync(0xffffffffu, p, o);
      if (ob > best || (ob == best && op < p)) { best = ob; p = op; }
    }
    if (!((float)best > rem)) {
      float left = 0;      // (FP32: the FP64 unit is slow, and a threshold is compared)
      for (int j = lane; j < qb; j += 32) left += fmaxf(0.f, (float)nr[j]);
      left = warp_sum_r(left);
      if (!(left > rem)) break;
      if constexpr (sizeof(R) == 4) {
        // many columns of like size: rounding noise, or aligned ones?  (Noise of that size moves
        // the singular values as much: up to two thirds of eps for half of it.)
        if (best <= 0.25f * rem && left >= 8.0f * best && left <= check) {
          if (left_norm2(C, ld, qa, qb, nr, red) <= (16.0f / 9.0f) * rem) break;
          check = 0.9f * left;
        }
      }
    }
    const R rs = rsqrt_of(best), ib = rcp_of(best);
    const Cx<R>* cp = C + p * ld;
    // kGL lanes a column: a warp in complex64, eight lanes in complex128 (an FP64 instruction
    // costs the same whatever the number of columns it serves)
    for (int jb = warp * kCPW; jb < qb; jb += nw * kCPW) {
      const int j = jb + lane / kGL, gl = lane % kGL;
      const bool in = j < qb, act = in && j != p && nr[in ? j : 0] >= 0;
      Cx<R>* cj = C + (act ? j : 0) * ld;
      Cx<R> d(0, 0);
      if (act)
        for (int i = gl; i < qa; i += kGL) cfma_conj(d, cp[i], cj[i]);
      for (int o = kGL / 2; o > 0; o >>= 1) d += shfl_xor(d, o);
      const Cx<R> be = -(ib * d);
      R acc = 0;
      if (act)
        for (int i = gl; i < qa; i += kGL) {
          Cx<R> v = cj[i];
          cfma(v, be, cp[i]);
          cj[i] = v;
          acc = fma(v.re, v.re, fma(v.im, v.im, acc));
        }
      for (int o = kGL / 2; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
      if (in && gl == 0) {
        nx[j] = act ? acc : R(-1);
        rk[j] = act ? rs * conj(d) : Cx<R>(j == p ? best * rs : R(0), R(0));
      }
    }
    // the row of the step before into the storage of its pivot column (read by nobody now)
    if (kq > 0 && warp == nw - 1) {
      const Cx<R>* rp = rbuf + ((kq & 1) ^ 1) * g.QCAP;
      Cx<R>* dst = C + slot[kq - 1] * ld;
      for (int j = lane; j < qb; j += 32) dst[j] = rp[j];
    }
    if (threadIdx.x == 0) slot[kq] = p;
    __syncthreads();
  }
  if (kq > 0) {
    const Cx<R>* rp = rbuf + ((kq & 1) ^ 1) * g.QCAP;
    Cx<R>* dst = C + slot[kq - 1] * ld;
    for (int j = threadIdx.x; j < qb; j += blockDim.x) dst[j] = rp[j];
  }
  // ---- 2. one-sided Jacobi on the kq columns (length qb) of L ------------------------------
  const int me = kq + (kq & 1);               // even number of positions (one dummy if odd)
  // one group of GW lanes per column pair: whole warps while there are at most as many
  // pairs as warps, half warps beyond (every pair of a round in one pass); in complex128 as
  // many pairs to a warp as keep four warps busy, one a scheduler's FP64 unit
  int GW = (me / 2 <= nw) ? 32 : 16;
  if (sizeof(R) == 8)
    while (GW > 4 && me / 2 * GW > 128) GW >>= 1;
  const int gpw = 32 / GW;                    // groups per warp
  for (int sweep = 0; sweep < 40; ++sweep) {
    __syncthreads();
    if (threadIdx.x == 0) s_rot = s_gg = s_t = 0;
    // squared column norms, exact at the start of every sweep and carried through its
    // rounds by the rotation's own update (a rotation by tan t of the pair (p, q) with
    // <p, q> = g maps |p|^2 to |p|^2 - t |g| and |q|^2 to |q|^2 + t |g|), so a pair's test
    // needs only the inner product
    for (int j = warp; j < kq; j += nw) {
      const Cx<R>* cj = C + slot[j] * ld;
      R acc = 0;
      for (int i = lane; i < qb; i += 32) acc += abs2(cj[i]);
      acc = warp_sum_r(acc);
      if (lane == 0) sig[j] = acc;
    }
    __syncthreads();
    for (int round = 0; round < me - 1; ++round) {
      // the loop bound is uniform over the warp, so every lane reaches every shuffle
      for (int pb = warp * gpw; pb < me / 2; pb += nw * gpw) {
        const int pr = pb + lane / GW, gl = lane % GW;
        const int p0 = pr, p1 = me - 1 - pr;
        int ip = p0 == 0 ? 0 : p0 - 1 + round, iq = p1 - 1 + round;
        if (p0 != 0) ip = (ip >= me - 1 ? ip - (me - 1) : ip) + 1;
        iq = (iq >= me - 1 ? iq - (me - 1) : iq) + 1;
        const bool live = pr < me / 2 && ip < kq && iq < kq;
        if (ip > iq) { const int tmp = ip; ip = iq; iq = tmp; }
        Cx<R>* cp = C + (live ? slot[ip] : 0) * ld;
        Cx<R>* cq = C + (live ? slot[iq] : 0) * ld;
        const R al = live ? sig[ip] : R(1), be = live ? sig[iq] : R(1);
        Cx<R> ga(0, 0);
        // (complex64, a warp a pair: the two columns stay in registers for the rotation)
        constexpr int NR = 5;
        const bool reg = sizeof(R) == 4 && GW == 32 && qb <= 32 * NR;
        Cx<float> xr[NR], yr[NR];
        if (reg) {
          if constexpr (sizeof(R) == 4) {
#pragma unroll
            for (int r = 0; r < NR; ++r) {
              const bool in = live && lane + 32 * r < qb;
              xr[r] = in ? cp[lane + 32 * r] : Cx<float>(0.f, 0.f);
              yr[r] = in ? cq[lane + 32 * r] : Cx<float>(0.f, 0.f);
              cfma_conj(ga, xr[r], yr[r]);
            }
          }
        } else if (live) {
          for (int i = gl; i < qb; i += GW) cfma_conj(ga, cp[i], cq[i]);
        }
        ga = group_sum(ga, GW);
        JacobiRotation<R> rot;
        if (rot.needed(al, be, ga, Tiny<R>::jac2) && live && al >= thr && be >= thr) {
          rot.angle(al, be);
          const R cs = rot.cs;
          const Cx<R> sne = rot.sne, snc = conj(sne);
          if (gl == 0) {
            if (rot.gg > Tiny<R>::quad) {
              s_rot = 1;
            } else {
              atomicMax(&s_gg, __float_as_int(rot.gg));      // (nonnegative floats order as integers)
              atomicMax(&s_t, __float_as_int(fabsf(rot.t)));
            }
            sig[ip] = fmax(R(0), al - rot.dn);
            sig[iq] = be + rot.dn;
          }
          if (reg) {
            if constexpr (sizeof(R) == 4) {
#pragma unroll
              for (int r = 0; r < NR; ++r)
                if (lane + 32 * r < qb) {
                  Cx<float> nx = cs * xr[r], ny = cs * yr[r];
                  cfma(nx, -snc, yr[r]);
                  cfma(ny, sne, xr[r]);
                  cp[lane + 32 * r] = nx;
                  cq[lane + 32 * r] = ny;
                }
            }
          } else {
            for (int i = gl; i < qb; i += GW) {
              const Cx<R> x = cp[i], y = cq[i];
              Cx<R> nx = cs * x, ny = cs * y;
              cfma(nx, -snc, y);
              cfma(ny, sne, x);
              cp[i] = nx;
              cq[i] = ny;
            }
          }
        }
      }
      __syncthreads();
    }
    if (s_rot == 0 && rotations_done(__int_as_float(s_gg), __int_as_float(s_t), Tiny<R>::jac2)) break;
  }
  // singular values, ordering, truncation
  for (int j = warp; j < kq; j += nw) {
    const Cx<R>* cj = C + slot[j] * ld;
    R acc = 0;
    for (int i = lane; i < qb; i += 32) acc += abs2(cj[i]);
    acc = warp_sum_r(acc);
    if (lane == 0) sig[j] = sqrt(acc);
  }
  if (threadIdx.x == 0) s_keep = 0;
  __syncthreads();
  for (int j = threadIdx.x; j < kq; j += blockDim.x) {
    int rk = 0;
    R smax = 0;
    for (int l = 0; l < kq; ++l) {
      rk += (sig[l] > sig[j] || (sig[l] == sig[j] && l < j)) ? 1 : 0;
      smax = fmax(smax, sig[l]);
    }
    order[rk] = j;
    // (a column below thr was left unrotated and need not be orthogonal to the others: at eps
    // below the rounding noise this is what ends the expansion)
    if (rk < g.r_max && sig[j] > R(eps) * smax && sig[j] * sig[j] > R(1.01) * thr) atomicMax(&s_keep, rk + 1);
  }
  __syncthreads();
  const int keep = s_keep;
  if (threadIdx.x == 0) {
    newrank[a] = keep;
    newrank[b] = keep;
  }
  Cx<R>* Ta = Tx + (long long)a * g.QCAP * g.r_max;   // column-major (ld QCAP)
  Cx<R>* Tb = Tx + (long long)b * g.QCAP * g.r_max;
  // balanced split, four columns of T_a per thread and pass over a row of C
  for (int e = threadIdx.x; e < qa * ((keep + 3) / 4); e += blockDim.x) {
    const int i = e % qa, j0 = (e / qa) * 4;
    Cx<R> acc[4];
    const Cx<R>* l[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      acc[u] = Cx<R>(0, 0);
      l[u] = C + slot[order[min(j0 + u, keep - 1)]] * ld;
    }
#pragma unroll 4
    for (int j = 0; j < qb; ++j) {
      const Cx<R> c = Cg[(long long)j * qa + i];
#pragma unroll
      for (int u = 0; u < 4; ++u) cfma(acc[u], c, l[u][j]);
    }
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (j0 + u < keep) {
        const R sg = sig[order[j0 + u]];
        Ta[(long long)(j0 + u) * g.QCAP + i] = (R(1) / (sg * sqrt(scale * sg))) * acc[u];
      }
  }
  for (int e = threadIdx.x; e < qb * keep; e += blockDim.x) {
    const int i = e % qb, j = e / qb;
    const R f = sqrt(scale / sig[order[j]]);
    Tb[(long long)j * g.QCAP + i] = f * conj(C[slot[order[j]] * ld + i]);
  }
}

// Recompression, step 3, for the nodes u = list[blockIdx.y]: F'_u = Q_u T_u (sz(u) x kr,
// column-major; T_u itself on the dense path) into the node's region of the scratch
// buffer Fs, one kCT x kCT tile per CTA (blockIdx.x), the k chunks of Q_u and T_u staged
// with coalesced loads; recompress_copy then moves it into G_F (Q_u is read from G_F
// until every tile is done).  The layer's last recompression, when it covers every node,
// writes the factor store and its ranks directly (Fs, off, rank_out).
template <typename R>
__global__ void __launch_bounds__(256) recompress_gemm(Geo g, const Cx<R>* __restrict__ G_F,
                                                       const int* __restrict__ qcols, const int* __restrict__ qmode,
                                                       const Cx<R>* __restrict__ Tx, const int* __restrict__ newrank,
                                                       Cx<R>* __restrict__ Fs, const long long* __restrict__ off,
                                                       int* __restrict__ rank_out) {
  pdl_begin();
  constexpr int kCT = core_tile_edge<R>(), U = kCT / 16;
  __shared__ Cx<R> Qs[kCK][kCT + 1], Ts[kCK][kCT + 1];
  const int u = g.list[blockIdx.y];
  const int s = g.sz[u], qc = qcols[u], kr = newrank[u];
  if (rank_out && blockIdx.x == 0 && threadIdx.x == 0) rank_out[u] = kr;
  const int ni = (s + kCT - 1) / kCT, nj = (kr + kCT - 1) / kCT;
  if ((int)blockIdx.x >= ni * nj) return;
  const int ti = blockIdx.x % ni, tj = blockIdx.x / ni;
  const Cx<R>* Qu = G_F + g.gfo[u];
  const Cx<R>* T = Tx + (long long)u * g.QCAP * g.r_max;
  Cx<R>* S = Fs + off[u];
  if (qmode[u]) {
    for (int e = threadIdx.x; e < kCT * kCT; e += blockDim.x) {
      const int i = ti * kCT + e % kCT, j = tj * kCT + e / kCT;
      if (i < s && j < kr) S[(long long)j * s + i] = T[(long long)j * g.QCAP + i];
    }
    return;
  }
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  Cx<R> acc[U][U];
  for (int a = 0; a < U; ++a)
    for (int b = 0; b < U; ++b) acc[a][b] = Cx<R>(0, 0);
  for (int k0 = 0; k0 < qc; k0 += kCK) {
    for (int e = threadIdx.x; e < kCK * kCT; e += blockDim.x) {
      const int r = e % kCT, kq = e / kCT;          // Q: consecutive threads, consecutive rows
      const int i = ti * kCT + r, k = k0 + kq;
      Qs[kq][r] = (i < s && k < qc) ? Qu[(long long)k * s + i] : Cx<R>(0, 0);
      const int kt = e % kCK, cc = e / kCK;         // T: consecutive threads, consecutive k
      const int j = tj * kCT + cc, k2 = k0 + kt;
      Ts[kt][cc] = (j < kr && k2 < qc) ? T[(long long)j * g.QCAP + k2] : Cx<R>(0, 0);
    }
    __syncthreads();
#pragma unroll 4
    for (int kk = 0; kk < kCK; ++kk)
#pragma unroll
      for (int a = 0; a < U; ++a)
#pragma unroll
        for (int b = 0; b < U; ++b) cfma(acc[a][b], Qs[kk][ty + 16 * a], Ts[kk][tx + 16 * b]);
    __syncthreads();
  }
  for (int a = 0; a < U; ++a)
    for (int b = 0; b < U; ++b) {
      const int i = ti * kCT + ty + 16 * a, j = tj * kCT + tx + 16 * b;
      if (i < s && j < kr) S[(long long)j * s + i] = acc[a][b];
    }
}

template <typename R>
__global__ void recompress_copy(Geo g, const Cx<R>* __restrict__ Fs, const int* __restrict__ newrank,
                                Cx<R>* __restrict__ G_F, int* __restrict__ G_rank) {
  pdl_begin();
  const int u = g.list[blockIdx.x];
  const int s = g.sz[u], kr = newrank[u];
  const Cx<R>* S = Fs + g.gfo[u];
  Cx<R>* F = G_F + g.gfo[u];
  for (int e = threadIdx.x; e < s * kr; e += blockDim.x) F[e] = S[e];
  if (threadIdx.x == 0) G_rank[u] = kr;
}

// T~_m into the factor store (leaf padding zeroed, factors truncated to r_max columns): the
// first nlb blocks store the leaves, the others the factor of node 2 + blockIdx.x - nlb (none
// of them when the recompression has stored the factors).
template <typename R>
__global__ void store_layer(Geo g, int nlb, const Cx<R>* __restrict__ G_leaf, const Cx<R>* __restrict__ G_F,
                            const int* __restrict__ G_rank, Cx<R>* __restrict__ dst, const long long* __restrict__ off,
                            int* __restrict__ rank_dst) {
  pdl_begin();
  if ((int)blockIdx.x < nlb) {
    const int lf = g.leaf;
    const int tot = (1 << g.L) * lf * lf;
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < tot; e += nlb * blockDim.x) {
      const int lam = (1 << g.L) + e / (lf * lf);
      const int r = e % (lf * lf);
      const int a = r % lf, b = r / lf, s = g.sz[lam];
      dst[e] = (a < s && b < s) ? G_leaf[e] : Cx<R>(0, 0);
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) { rank_dst[0] = 0; rank_dst[1] = 0; }
    return;
  }
  const int v = 2 + (int)blockIdx.x - nlb;
  const int s = g.sz[v], r = G_rank[v];
  const Cx<R>* F = G_F + g.gfo[v];
  for (int e = threadIdx.x; e < s * r; e += blockDim.x) dst[off[v] + e] = F[e];
  if (threadIdx.x == 0) rank_dst[v] = r;
}

}  // namespace

// ---------------------------------------------------------------------------------------
struct SetupWork {
  int KCAP = 0, WCAP = 0, QCAP = 0, dense_max = 0;
  long long gfo_total = 0;   // entries of one G factor buffer
  std::vector<long long> sfo, gfo, qro, rbo;
  std::vector<int> rowleaf, cap;
  // node lists of the recompression launches: for depth step d, the nodes of the
  // non-deferred depths below d (big_nodes[d] .. big_nodes[d+1]) and their left siblings
  // (big_pairs), then the nodes of the deferred depths (small_*) and all nodes (all_*)
  std::vector<int> lists;
  std::vector<int> big_nodes_off, big_pairs_off;
  int small_nodes_off = 0, small_nodes = 0, small_pairs_off = 0, small_pairs = 0;
  int all_nodes_off = 0, all_nodes = 0, all_pairs_off = 0, all_pairs = 0;
  long long* d_sfo = nullptr;
  long long* d_gfo = nullptr;
  long long* d_qro = nullptr;
  long long* d_rbo = nullptr;
  int* d_rowleaf = nullptr;
  int* d_cap = nullptr;
  int* d_lists = nullptr;
  void *S_F = nullptr, *G_leaf = nullptr, *G_F = nullptr, *G_F2 = nullptr;
  void *Y = nullptr, *W = nullptr, *Qr = nullptr, *PQ = nullptr, *M = nullptr, *Rb = nullptr;
  void *Tx = nullptr, *Cb = nullptr;
  int *S_rank = nullptr, *G_rank = nullptr, *qcols = nullptr, *qmode = nullptr, *newrank = nullptr;
};

void hsw_setup_free(hsweep_s* h) {
  if (!h->sw) return;
  SetupWork* w = h->sw;
  void* ptrs[] = {w->d_sfo, w->d_gfo, w->d_qro, w->d_rbo, w->d_rowleaf, w->d_cap, w->d_lists, w->S_F,
                  w->G_leaf, w->G_F, w->G_F2, w->Y, w->W, w->Qr, w->PQ, w->M, w->Rb, w->Tx, w->Cb, w->S_rank,
                  w->G_rank, w->qcols, w->qmode, w->newrank};
  for (void* p : ptrs) hsw_release(h, p);
  delete w;
  h->sw = nullptr;
}

static int depth_of_host(int v) { int d = 0; while ((2 << d) <= v) ++d; return d; }

static int setup_alloc(hsweep_s* h) {
  SetupWork* w = new (std::nothrow) SetupWork();
  if (!w) return HSWEEP_ERR_OOM;
  h->sw = w;
  const size_t es = h->fac_elem();
  const int nn = h->nnodes, L = h->L;
  w->KCAP = h->r_max + 1;
  w->WCAP = h->r_max + w->KCAP;
  // A depth is deferred when the largest core its blocks can reach at the end of a layer,
  // min(rows, depth x KCAP) (every depth step above appends at most KCAP columns), fits the
  // Jacobi SVD's shared memory; its blocks are recompressed once per layer.  The other
  // depths are recompressed after every depth step (at most WCAP columns).
  const size_t smem_cap = 227 * 1024 - 8192;
  const int qlim = (int)std::sqrt((double)(smem_cap / es));
  auto deferred_core = [&](int d) { return std::min(h->tree.maxsz(d), d * w->KCAP); };
  auto small_depth = [&](int d) { return deferred_core(d) <= qlim; };
  w->QCAP = w->WCAP;
  w->dense_max = es == sizeof(c64) ? kDenseRows : 0;
  for (int d = 1; d <= L; ++d)
    if (small_depth(d)) w->QCAP = std::max(w->QCAP, deferred_core(d));
  // (node by node: n = 257 or 513 has depths with blocks of 128 and of 129 rows)
  for (int v = 2; v < nn; ++v)
    if (h->tree.sz[v] <= w->dense_max) w->QCAP = std::max(w->QCAP, h->tree.sz[v]);
  w->sfo.assign(nn, 0);
  w->gfo.assign(nn, 0);
  w->qro.assign(nn, 0);
  w->rbo.assign(nn, 0);
  w->cap.assign(nn, 0);
  long long so = 0, go = 0, qo = 0, ro = 0;
  for (int v = 2; v < nn; ++v) {
    const int d = depth_of_host(v), sv = h->tree.sz[v];
    const int cv = small_depth(d) ? d * w->KCAP : w->WCAP;
    w->cap[v] = cv;
    w->sfo[v] = so; so += (long long)sv * w->KCAP;
    w->gfo[v] = go; go += (long long)sv * cv;
    w->qro[v] = qo; qo += (long long)cv * w->KCAP;
    w->rbo[v] = ro; ro += (long long)(sv <= w->dense_max ? sv : std::min(sv, cv)) * cv;
  }
  // recompression lists
  w->lists.clear();
  w->big_nodes_off.assign(L + 1, 0);
  w->big_pairs_off.assign(L + 1, 0);
  for (int d = 0; d < L; ++d) {
    w->big_nodes_off[d] = (int)w->lists.size();
    for (int v = 2; v < nn; ++v)
      if (depth_of_host(v) > d && !small_depth(depth_of_host(v))) w->lists.push_back(v);
  }
  w->big_nodes_off[L] = (int)w->lists.size();
  for (int d = 0; d < L; ++d) {
    w->big_pairs_off[d] = (int)w->lists.size();
    for (int v = 2; v < nn; v += 2)
      if (depth_of_host(v) > d && !small_depth(depth_of_host(v))) w->lists.push_back(v);
  }
  w->big_pairs_off[L] = (int)w->lists.size();
  w->small_nodes_off = (int)w->lists.size();
  for (int v = 2; v < nn; ++v)
    if (small_depth(depth_of_host(v))) w->lists.push_back(v);
  w->small_nodes = (int)w->lists.size() - w->small_nodes_off;
  w->small_pairs_off = (int)w->lists.size();
  for (int v = 2; v < nn; v += 2)
    if (small_depth(depth_of_host(v))) w->lists.push_back(v);
  w->small_pairs = (int)w->lists.size() - w->small_pairs_off;
  w->all_nodes_off = (int)w->lists.size();
  for (int v = 2; v < nn; ++v) w->lists.push_back(v);
  w->all_nodes = nn - 2;
  w->all_pairs_off = (int)w->lists.size();
  for (int v = 2; v < nn; v += 2) w->lists.push_back(v);
  w->all_pairs = (nn - 2) / 2;

  w->rowleaf.assign(h->n, 0);
  for (int lam = h->nleaves; lam < 2 * h->nleaves; ++lam)
    for (int i = 0; i < h->tree.sz[lam]; ++i) w->rowleaf[h->tree.lo[lam] + i] = lam;
  const long long lf2 = (long long)h->nleaves * h->leaf * h->leaf;
  const long long ntau = std::max(1, h->nleaves / 2);
  int rc;
#define A(p, bytes) do { rc = hsw_alloc(h, (void**)&(p), (size_t)(bytes)); if (rc) return rc; } while (0)
  A(w->d_sfo, nn * sizeof(long long));
  A(w->d_gfo, nn * sizeof(long long));
  A(w->d_qro, nn * sizeof(long long));
  A(w->d_rbo, nn * sizeof(long long));
  A(w->d_rowleaf, h->n * sizeof(int));
  A(w->d_cap, nn * sizeof(int));
  A(w->d_lists, std::max<size_t>(1, w->lists.size()) * sizeof(int));
  A(w->G_leaf, lf2 * es);
  A(w->S_F, std::max(so, 1LL) * es);
  A(w->G_F, std::max(go, 1LL) * es);
  A(w->G_F2, std::max(go, 1LL) * es);
  w->gfo_total = std::max(go, 1LL);
  A(w->Y, (long long)h->n * w->KCAP * es);
  A(w->W, (long long)h->n * w->KCAP * es);
  A(w->Qr, std::max(qo, 1LL) * es);
  A(w->PQ, ntau * 2 * w->KCAP * w->KCAP * es);
  A(w->M, ntau * 4 * w->KCAP * w->KCAP * es);
  A(w->Rb, std::max(ro, 1LL) * es);
  A(w->Tx, (long long)nn * w->QCAP * h->r_max * es);
  A(w->Cb, (long long)(nn / 2) * w->QCAP * w->QCAP * es);
  A(w->S_rank, nn * sizeof(int));
  A(w->G_rank, nn * sizeof(int));
  A(w->qcols, nn * sizeof(int));
  A(w->qmode, nn * sizeof(int));
  A(w->newrank, nn * sizeof(int));
#undef A
  HSW_CUDA(cudaMemcpyAsync(w->d_sfo, w->sfo.data(), nn * sizeof(long long), cudaMemcpyHostToDevice, h->stream));
  HSW_CUDA(cudaMemcpyAsync(w->d_gfo, w->gfo.data(), nn * sizeof(long long), cudaMemcpyHostToDevice, h->stream));
  HSW_CUDA(cudaMemcpyAsync(w->d_qro, w->qro.data(), nn * sizeof(long long), cudaMemcpyHostToDevice, h->stream));
  HSW_CUDA(cudaMemcpyAsync(w->d_rbo, w->rbo.data(), nn * sizeof(long long), cudaMemcpyHostToDevice, h->stream));
  HSW_CUDA(cudaMemcpyAsync(w->d_cap, w->cap.data(), nn * sizeof(int), cudaMemcpyHostToDevice, h->stream));
  HSW_CUDA(cudaMemcpyAsync(w->d_rowleaf, w->rowleaf.data(), h->n * sizeof(int), cudaMemcpyHostToDevice, h->stream));
  if (!w->lists.empty())
    HSW_CUDA(cudaMemcpyAsync(w->d_lists, w->lists.data(), w->lists.size() * sizeof(int), cudaMemcpyHostToDevice,
                             h->stream));
  HSW_CUDA(cudaMemsetAsync(w->S_rank, 0, nn * sizeof(int), h->stream));
  HSW_CUDA(cudaMemsetAsync(w->G_rank, 0, nn * sizeof(int), h->stream));
  // the host vectors above are read by the asynchronous copies: keep them until the copies ran
  HSW_CUDA(cudaStreamSynchronize(h->stream));
  return HSWEEP_OK;
}

template <typename R>
static int factor_impl(hsweep_s* h) {
  SetupWork* w = h->sw;
  const size_t es = sizeof(Cx<R>);
  Geo g;
  g.n = h->n; g.L = h->L; g.leaf = h->leaf; g.nnodes = h->nnodes; g.r_max = h->r_max;
  g.KCAP = w->KCAP; g.WCAP = w->WCAP; g.QCAP = w->QCAP; g.dense_max = w->dense_max;
  g.cap_max = *std::max_element(w->cap.begin(), w->cap.end());
  g.lo = h->d_lo; g.sz = h->d_sz; g.rowleaf = w->d_rowleaf; g.sfo = w->d_sfo; g.gfo = w->d_gfo;
  g.cap = w->d_cap; g.qro = w->d_qro; g.rbo = w->d_rbo; g.list = w->d_lists;
  cudaStream_t st = h->stream;
  Cx<R>* fac = reinterpret_cast<Cx<R>*>(h->d_fac);
  Cx<R>* S_F = (Cx<R>*)w->S_F;
  Cx<R>* G_leaf = (Cx<R>*)w->G_leaf;
  Cx<R>* G_F = (Cx<R>*)w->G_F;
  Cx<R>* G_F2 = (Cx<R>*)w->G_F2;
  Cx<R>* Y = (Cx<R>*)w->Y;
  Cx<R>* Wv = (Cx<R>*)w->W;
  Cx<R>* Qr = (Cx<R>*)w->Qr;
  Cx<R>* PQ = (Cx<R>*)w->PQ;
  Cx<R>* M = (Cx<R>*)w->M;
  Cx<R>* Rb = (Cx<R>*)w->Rb;
  Cx<R>* Tx = (Cx<R>*)w->Tx;
  const int L = h->L, nn = h->nnodes, KCAP = w->KCAP, QCAP = w->QCAP;
  const size_t core_smem = (size_t)(2 * KCAP) * (2 * KCAP) * es + 32 * sizeof(R) + (2 * KCAP + 1) * sizeof(int) + 16;
  // QR: norms and positions, then as many entries of F_u as fit (226 KB in all)
  const size_t qr_base = qr_tables<R>(g.cap_max);
  const int qs_entries = qr_base < 226 * 1024 ? (int)((226 * 1024 - qr_base) / es) : 0;
  const size_t qr_smem = qr_base + (size_t)qs_entries * es;
  const SvdPlan<R> svd(QCAP, h->eps_H);
  // one shared-memory carveout for every kernel of the layer loop, so that consecutive
  // launches do not reconfigure the SMs' L1/shared split
  {
    const void* ks[] = {(const void*)schur_layer<R>,
                        (const void*)tsmm_reduce<R>, (const void*)tsmm_expand<R>, (const void*)core_dots<R>,
                        (const void*)core_inverse<R>, (const void*)woodbury_form<R>, (const void*)woodbury_append<R>,
                        (const void*)qr_mgs<R>, (const void*)svd_jacobi<R>, (const void*)recompress_gemm<R>,
                        (const void*)recompress_copy<R>, (const void*)store_layer<R>, (const void*)core_product_cc<R>};
    for (const void* k : ks)
      HSW_CUDA(cudaFuncSetAttribute(k, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared));
  }
  // (four KCAP x KCAP blocks and tables: also holds the three blocks of core_inverse_block)
  HSW_CUDA(cudaFuncSetAttribute(core_inverse<R>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)core_smem));
  HSW_CUDA(cudaFuncSetAttribute(core_inverse_block, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)core_smem));
  HSW_CUDA(cudaFuncSetAttribute(core_inverse_block, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared));
  HSW_CUDA(cudaFuncSetAttribute(qr_mgs<R>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)qr_smem));
  HSW_CUDA(cudaFuncSetAttribute(svd_jacobi<R>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)svd.smem));
  if (core_smem > 227 * 1024 || qr_smem > 227 * 1024 || svd.smem > 227 * 1024)
    return HSWEEP_ERR_ARG;

  // Autotuning of the core products (step 2a), complex64 only: on layer tune_m, the first
  // launch of each kind (0: the recompressions after a depth step, 1: the once-per-layer
  // recompression) runs both kernels, timed with CUDA events, and the faster one serves that
  // kind of launch from then on; before it, and in complex128, the CUDA-core kernel runs.
  const int tune_m = h->n / 2;
  constexpr int kCT = core_tile_edge<R>();
  const int core_tiles = ((QCAP + kCT - 1) / kCT) * ((QCAP + kCT - 1) / kCT);
  const int gemm_tiles = ((h->tree.maxsz(1) + kCT - 1) / kCT) * ((h->r_max + kCT - 1) / kCT);
  Cx<R>* Cb = (Cx<R>*)w->Cb;
  int m_cur = 0;
  auto core_product = [&](const Geo& gp, int np_list, int kind) -> int {
    const dim3 grid(core_tiles, np_list);
    const bool f32 = sizeof(R) == 4;
    auto run = [&](int mode) -> cudaError_t {
      if constexpr (sizeof(R) == 4) {
        if (mode == 1) {
          return pdl_launch(core_product_tc, grid, 256, 0, st, gp, (const Cx<float>*)Rb, w->qcols, w->G_rank,
                            (Cx<float>*)Cb);
        }
      }
      return pdl_launch(core_product_cc<R>, grid, 256, 0, st, gp, Rb, w->qcols, w->G_rank, Cb);
    };
    if (h->opt.core_kernel > 0) {          // fixed by the caller
      HSW_CUDA(run(f32 && h->opt.core_kernel == 2 ? 1 : 0));
      h->nlaunch += 1;
      return HSWEEP_OK;
    }
    if (f32 && h->core_mode[kind] < 0 && m_cur == tune_m) {
      cudaEvent_t ev[3];
      for (auto& e : ev) HSW_CUDA(cudaEventCreate(&e));
      HSW_CUDA(cudaEventRecord(ev[0], st));
      HSW_CUDA(run(0));
      HSW_CUDA(cudaEventRecord(ev[1], st));
      HSW_CUDA(run(1));
      HSW_CUDA(cudaEventRecord(ev[2], st));
      HSW_CUDA(cudaEventSynchronize(ev[2]));
      float t0 = 0, t1 = 0;
      HSW_CUDA(cudaEventElapsedTime(&t0, ev[0], ev[1]));
      HSW_CUDA(cudaEventElapsedTime(&t1, ev[1], ev[2]));
      for (auto& e : ev) cudaEventDestroy(e);
      h->core_ms[kind][0] = t0;
      h->core_ms[kind][1] = t1;
      h->core_mode[kind] = t1 < t0 ? 1 : 0;
      h->nlaunch += 2;
      return HSWEEP_OK;
    }
    HSW_CUDA(run(f32 && h->core_mode[kind] == 1 ? 1 : 0));
    h->nlaunch += 1;
    return HSWEEP_OK;
  };

  // QR (or the dense path), the cores, their SVD and the new factors, for nn_list nodes
  // whose list starts at node_off and their np_list left siblings at pair_off
  auto recompress = [&](int node_off, int nn_list, int pair_off, int np_list, int kind, Cx<R>* store = nullptr,
                        int* store_rank = nullptr) -> int {
    if (nn_list <= 0) return HSWEEP_OK;
    Geo gl = g;
    gl.list = w->d_lists + node_off;
    HSW_CUDA(pdl_launch(qr_mgs<R>, dim3(nn_list), 1024, qr_smem, st, gl, G_F, w->G_rank, Rb, w->qcols, w->qmode, qs_entries));
    Geo gp = g;
    gp.list = w->d_lists + pair_off;
    int rc = core_product(gp, np_list, kind);
    if (rc) return rc;
    HSW_CUDA(pdl_launch(svd_jacobi<R>, dim3(np_list), 1024, svd.smem, st, gp, h->eps_H, Cb, w->qcols, Tx, w->newrank, svd.entries, svd.thr, svd.rem));
    if (store) {
      HSW_CUDA(pdl_launch(recompress_gemm<R>, dim3(gemm_tiles, nn_list), 256, 0, st, gl, G_F, w->qcols, w->qmode, Tx, w->newrank, store, h->d_off, store_rank));
      h->nlaunch += 3;
      return HSWEEP_OK;
    }
    HSW_CUDA(pdl_launch(recompress_gemm<R>, dim3(gemm_tiles, nn_list), 256, 0, st, gl, G_F, w->qcols, w->qmode, Tx, w->newrank, G_F2, w->d_gfo, (int*)nullptr));
    HSW_CUDA(pdl_launch(recompress_copy<R>, dim3(nn_list), kBlk, 0, st, gl, G_F2, w->newrank, G_F, w->G_rank));
    h->nlaunch += 4;
    return HSWEEP_OK;
  };

  for (int m = 0; m < h->n; ++m) {
    NvtxRange range("setup layer");
    m_cur = m;
    const Cx<R>* Tprev = m > 0 ? fac + (long long)(m - 1) * h->layer_stride : nullptr;
    const int* rprev = m > 0 ? h->d_rank + (long long)(m - 1) * nn : nullptr;
    HSW_CUDA(pdl_launch(schur_layer<R>, dim3(h->nleaves + nn - 2, nn > 2 ? 8 : 1), kBlk, 0, st, g, m, h->d_diag_m,
                        h->d_east_m, h->d_north_m, Tprev, h->d_off, rprev, S_F, w->S_rank, G_leaf, w->G_rank,
                        h->d_status));
    h->nlaunch += 1;
    for (int d = L - 1; d >= 0; --d) {
      const int n_below2 = (d + 2 <= L) ? (1 << (L + 1)) - (1 << (d + 2)) : 0;
      const int n_below1 = (1 << (L + 1)) - (1 << (d + 1));
      const int ntau_d = 1 << d;
      if (n_below2 > 0) {
        HSW_CUDA(pdl_launch(tsmm_reduce<R>, dim3(n_below2, (KCAP + 7) / 8), kBlk, 0, st, g, d, G_F, w->G_rank, S_F, w->S_rank, Qr));
        h->nlaunch += 1;
      }
      HSW_CUDA(pdl_launch(tsmm_expand<R>, dim3(div_up(h->n, 32), (KCAP + 3) / 4), kBlk, 0, st, g, d, G_leaf, G_F,
                          w->G_rank, S_F, w->S_rank, Qr, Y));
      h->nlaunch += 1;
      HSW_CUDA(pdl_launch(core_dots<R>, dim3(2 * ntau_d, std::max(8, 64 / (2 * ntau_d))), kBlk, 0, st, g, d, S_F, w->S_rank, Y, PQ));
      h->nlaunch += 1;
      if constexpr (sizeof(R) == 4)
        HSW_CUDA(pdl_launch(core_inverse_block, dim3(ntau_d), 32 * kCoreWarps, core_smem, st, g, d, m, w->S_rank, PQ, M, h->d_status));
      else
        HSW_CUDA(pdl_launch(core_inverse<R>, dim3(ntau_d), 1024, core_smem, st, g, d, m, w->S_rank, PQ, M, h->d_status));
      h->nlaunch += 1;
      HSW_CUDA(pdl_launch(woodbury_form<R>, dim3(div_up(h->n, 32), (KCAP + 3) / 4), 128, 0, st, g, d, w->S_rank, Y, M, Wv,
                          G_F, w->G_rank));
      h->nlaunch += 1;
      HSW_CUDA(pdl_launch(woodbury_append<R>, dim3(n_below1), kBlk, 0, st, g, d, w->S_rank, Y, Wv, G_F, w->G_rank, G_leaf));
      h->nlaunch += 1;
      // the blocks of the non-deferred depths that this depth step changed
      int rc = recompress(w->big_nodes_off[d], w->big_nodes_off[d + 1] - w->big_nodes_off[d], w->big_pairs_off[d],
                          w->big_pairs_off[d + 1] - w->big_pairs_off[d], 0);
      if (rc) return rc;
    }
    // the blocks of the deferred depths, once per layer, in their final form
    Cx<R>* store = fac + (long long)m * h->layer_stride;
    int* store_rank = h->d_rank + (long long)m * nn;
    const bool direct = nn > 2 && (h->strong_R > 0 || w->small_nodes == nn - 2);   // the last one covers every node
    {
      const bool last = direct && h->strong_R == 0;
      int rc = recompress(w->small_nodes_off, w->small_nodes, w->small_pairs_off, w->small_pairs, 1,
                          last ? store : nullptr, store_rank);
      if (rc) return rc;
    }
    if (h->strong_R > 0) {
      // strongly admissible T~_m (strong.cu), then one recompression of every sibling pair:
      // the expanded layout can carry more columns than a block has rows (small blocks,
      // blocks of rank below R); the recompression keeps the same matrix up to eps_H and
      // brings every rank to at most the block's dimensions, as the sweeps expect
      int rc = hsw_strong_project(h, m, G_F, w->G_rank, G_F2, w->d_gfo, w->gfo_total);
      if (rc) return rc;
      std::swap(G_F, G_F2);
      // the records of the strong sweep, from the exact strongly admissible factors
      rc = hsw_spack_layer(h, m, G_F, G_leaf, w->d_gfo);
      if (rc) return rc;
      rc = hsw_strong_slabs(h, m, G_F, G_leaf, w->d_gfo, w->G_rank);
      if (rc) return rc;
      rc = recompress(w->all_nodes_off, w->all_nodes, w->all_pairs_off, w->all_pairs, 1, direct ? store : nullptr,
                      store_rank);
      if (rc) return rc;
    }
    const int nlb = (int)std::min<long long>(64, div_up(h->leaf_entries, kBlk));
    HSW_CUDA(pdl_launch(store_layer<R>, dim3(direct ? nlb : nlb + nn - 2), kBlk, 0, st, g, nlb, G_leaf, G_F, w->G_rank, store,
                        h->d_off, store_rank));
    h->nlaunch += 1;
    HSW_CUDA(cudaGetLastError());
  }
  w->G_F = G_F;
  w->G_F2 = G_F2;
  return HSWEEP_OK;
}

int hsw_factor(hsweep_s* h) {
  if (!h->sw) {
    int rc = setup_alloc(h);
    if (rc) return rc;
  }
  if (h->prec == HSWEEP_FP64) return factor_impl<double>(h);
  return factor_impl<float>(h);
}
