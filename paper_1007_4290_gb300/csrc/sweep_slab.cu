// The apply z = M r of Algorithm 2.6 by thread-block clusters on dense-diagonal slabs.
//
// A cluster of C = 2^dC CTAs carries G right-hand sides through the 2n-1 dependent
// hmatvecs; CTA c owns the rows of the depth-dC tree node 2^dC + c (its slab, ns rows).
// T~_m restricted to a slab is stored dense, and of the factors only the ancestors' rows
// remain (depths 1..dC, the columns of all depths side by side):
//     y = D x + F q,   q_v = sum over the CTAs of the sibling subtree of F^t x .
// What bounds a step is its latency, not its arithmetic or its bytes: the 2n-1 steps are a
// chain, and a step is two small products around one exchange between the CTAs.  So the
// layout removes everything else from the chain:
//   - the dense diagonal replaces the tree below the slab: no reductions, barriers or
//     descriptor tables for the depths > dC.  It is also work that does not need the
//     exchange, so it runs while the partial sums travel;
//   - one flat loop over the columns of all depths, no per-depth tables: a layer needs the
//     dC column boundaries only;
//   - the exchange is one message per sum: st.async puts a partial sum into the shared memory
//     of the CTA that reads it and completes its bytes on that CTA's mbarrier.  No memory
//     round trip, no fence, no tags.  (A variant that left the sums at home, arrived with
//     release semantics and let the readers fetch them took 0.4 us a step longer: the
//     release waits for the step's own global stores.)
// A step has two block barriers (x complete; sums and D x complete) and one mbarrier wait.
//
// One step (layer m):
//   1. p = F^t x, warps over chunks of kKW columns (lane = columns x row subset), each sum
//      sent to the CTAs of the sibling subtree (slot = its column and sender);
//   2. D x, the same loop over the columns of D^t, while the messages travel;
//   3. wait for the received bytes of this step (known from the layer's columns), add the
//      contributions: q;
//   4. y = D x + F q, each lane a slice of the columns for RA rows, reduced so that every lane
//      ends with one (row, right-hand side), and the update of Algorithm 2.6 on that value in
//      registers.
// The receive buffer of step t is rewritten by messages of step t + 2; their sender waited
// for this CTA's messages of step t + 1, which were sent after step t was read.  (Every pair
// of CTAs exchanges at least one column in every step: empty blocks get a zero column.)
// Bulk copies bring the next layer's F (two stages) and D (two, or one when shared memory
// is short: D is free from the second barrier on).  The update's global inputs are copied
// one step ahead into shared memory.
//
// Clusters of 16 CTAs are at most seven at a time (one per GPC with 16 free SMs), and the
// receive buffer grows with G.  Where more teams fit side by side without clusters (n = 1023
// with 64 right-hand sides: eight teams of 16), the same kernel runs as a cooperative grid
// and exchanges tagged words through L2 (sweep_team.cu's protocol; L2X below).
//
// Measured (eps_H 1e-6), per step, against the team sweep of sweep_team.cu: complex64, n = 511,
// lens: 2.0 us with one right-hand side (5.0), 2.8 with 16 (5.6), 4.5 with 64 (7.5); n = 1023,
// random medium, the top ranks at 48: 2.9 with one (6.2), 5.3 with 16 (7.2), 8.4 with 64
// (12.4); complex128, n = 255, random, with four: 4.9 (8.6).  What a step takes is instruction latency: with one right-hand
// side 600 instructions a warp at one in four clocks and scheduler; with eight about 5 us of
// FP32 multiply-adds and shared-memory reads.  Not kept: two half-CTAs with four right-hand
// sides each on the same stages (register spills: 10.2 us against 8.0), and the paired FP32
// instruction in the tiles (77 % of the FP32 rate where plain multiply-adds reach 88 %).
#include <algorithm>
#include <cstdlib>
#include <type_traits>
#include "handle.h"
#include "sweep_common.cuh"
#include "tma.cuh"

namespace {

using namespace tma;
using namespace sweepc;

constexpr long long kWaitLimit = 1LL << 22;   // bounded waits

// Register tiles.  A lane multiplies A columns (steps 1, 2) by B right-hand sides; the eight
// of G = 8 are split over two lanes.  CL lanes side by side cover a chunk of kKW columns, the
// other lanes of the warp take every RL-th row.  Shared memory delivers 4 bytes a lane and
// clock whatever is broadcast, so an A x B tile costs 2 (A + B) clocks of loads and A B
// clocks of FP32 multiply-adds per row: 1 x 8 tiles are load-bound (18 against 8), 4 x 4 ones
// balanced.  In complex128 the FP64 unit is the bound: one column a lane and two row subsets,
// few additions to join them.
template <typename R, int G> struct Tile;
template <int G> struct Tile<float, G> {
  static constexpr int A = 4, CL = 4, B = G > 4 ? 4 : G;
};
template <int G> struct Tile<double, G> {
  static constexpr int A = 1, CL = 16, B = G;
};
constexpr int kKW = 16;       // columns per chunk, in both precisions

// acc += f x for B right-hand sides (in pairs, the FP32 instruction on two values costs as many
// moves as it saves), and their B values of a row
template <typename R, int B>
__device__ __forceinline__ void mac(Cx<R> (&s)[B], Cx<R> f, const Cx<R> (&x)[B]) {
#pragma unroll
  for (int g = 0; g < B; ++g) cfma(s[g], f, x[g]);
}
template <typename R, int B>
__device__ __forceinline__ void load_rhs(const Cx<R>* p, Cx<R> (&x)[B]) {
  if constexpr (sizeof(R) == 4 && B % 2 == 0) {
#pragma unroll
    for (int g = 0; g < B; g += 2) {
      const float4 v = *reinterpret_cast<const float4*>(p + g);
      x[g] = Cx<R>(v.x, v.y);
      x[g + 1] = Cx<R>(v.z, v.w);
    }
  } else {
#pragma unroll
    for (int g = 0; g < B; ++g) x[g] = p[g];
  }
}
// entries per row of F (or D) for w columns: a multiple of 8, odd in units of 64 bytes, so
// that the rows of a warp's access fall into different banks
template <typename R>
__host__ __device__ constexpr int slab_stride(int w) {
  constexpr int U = sizeof(R) == 4 ? 8 : 4;
  const int u = (w + U - 1) / U;
  return u == 0 ? 0 : (u | 1) * U;
}

// ---- cluster primitives ------------------------------------------------------------------
__device__ __forceinline__ unsigned mapa(unsigned addr, unsigned rank) {
  unsigned r;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// one value (8 or 16 bytes) into another CTA's shared memory; its bytes complete on that CTA's
// mbarrier.  No fence: the data and the signal travel together.
__device__ __forceinline__ void send(unsigned addr, Cx<float> v, unsigned bar) {
  asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v2.b32 [%0], {%1, %2}, [%3];" ::"r"(addr),
               "r"(__float_as_uint(v.re)), "r"(__float_as_uint(v.im)), "r"(bar)
               : "memory");
}
__device__ __forceinline__ void send(unsigned addr, Cx<double> v, unsigned bar) {
  asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v2.b64 [%0], {%1, %2}, [%3];" ::"r"(addr),
               "l"((u64)__double_as_longlong(v.re)), "l"((u64)__double_as_longlong(v.im)), "r"(bar)
               : "memory");
}
// two neighbouring complex64 values, 16-byte aligned
__device__ __forceinline__ void send2(unsigned addr, Cx<float> v, Cx<float> w, unsigned bar) {
  asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1, %2, %3, %4}, [%5];" ::"r"(addr),
               "r"(__float_as_uint(v.re)), "r"(__float_as_uint(v.im)), "r"(__float_as_uint(w.re)),
               "r"(__float_as_uint(w.im)), "r"(bar)
               : "memory");
}

// two tagged words (16 bytes); teams exchange through L2 in complex64 only
__device__ __forceinline__ void load_words(const Tagged<float>::W* p, Tagged<float>::W (&w)[2]) {
  const ulonglong2 t = __ldcg(reinterpret_cast<const ulonglong2*>(p));
  w[0] = t.x;
  w[1] = t.y;
}
__device__ __forceinline__ void store_words(Tagged<float>::W* p, Tagged<float>::W w0, Tagged<float>::W w1) {
  __stcg(reinterpret_cast<ulonglong2*>(p), make_ulonglong2(w0, w1));
}

template <typename R>
struct SlabArgs {
  int n, dC, C, nrhs, rsD, dbufs, Wcap, group0;
  long long N, cap;             // entries per (layer, slab) record
  const int* lo;
  const int* sz;
  const uchar4* meta;           // [C][n] end column of the depths 1..4
  const Cx<R>* pack;            // [n][C][cap]: D^t (ns x rsD), then F (ns x slab_stride(W))
  const Cx<R>* cpl;             // coupling between the layers, [n + 1][n], in the storage precision
  const c128* r;
  c128* z;
  Cx<R>* w;
  typename Tagged<R>::W* xch;   // L2 teams: tagged partial sums [2][teams][C][Wcap][G]
  int* status;
  long long wait_limit;         // iterations of the waits for other CTAs
  int withhold;                 // test only: this CTA never arrives (-1: none)
  unsigned o_F[2], o_D[2], o_x, o_q, o_p[2], o_y, o_bar, o_meta;
  unsigned o_in, o_inc;         // the update's inputs: r or w of every (row, rhs), couplings of every row
};

template <typename R, int G, int RA, int CS, int NT, bool L2X>
__global__ void __launch_bounds__(NT, G == 4 && NT == 256 ? 2 : 1) sweep_slab_kernel(SlabArgs<R> a) {
  extern __shared__ __align__(128) unsigned char sm[];
  constexpr int GS = vstride<R>(G);
  using TL = Tile<R, G>;
  constexpr int A = TL::A, CL = TL::CL, B = TL::B, GL = G / B, RL = 32 / (CL * GL), KW = kKW;
  constexpr int NW = NT / 32;
  constexpr int RG = 32 / (CS * GL);      // step 4: row groups per warp, RA rows each
  constexpr int VG = (sizeof(R) == 4 && G % 2 == 0) ? 2 : 1;    // right-hand sides per 16-byte word
  using T = Tagged<R>;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int n = a.n, dC = a.dC, C = a.C;
  const int c = blockIdx.x % C;
  const int g0 = (a.group0 + blockIdx.x / C) * G;
  const int gcount = min(G, a.nrhs - g0);
  const int lo_c = a.lo[C + c], ns = a.sz[C + c];
  const int nsteps = 2 * n - 1;

  Cx<R>* x = reinterpret_cast<Cx<R>*>(sm + a.o_x);
  Cx<R>* q = reinterpret_cast<Cx<R>*>(sm + a.o_q);
  Cx<R>* yl = reinterpret_cast<Cx<R>*>(sm + a.o_y);
  unsigned long long* bars = reinterpret_cast<unsigned long long*>(sm + a.o_bar);
  unsigned long long *barF = bars, *barD = bars + 2, *barX = bars + 4;
  volatile int* s_fail = reinterpret_cast<volatile int*>(bars + 6);

  if (tid == 0) {
    for (int b = 0; b < 2; ++b) {
      mbar_init(&barF[b], 1);
      mbar_init(&barD[b], 1);
      mbar_init(&barX[b], 1);
    }
    *s_fail = 0;
    fence_mbar_init();
  }
  uchar4* s_meta = reinterpret_cast<uchar4*>(sm + a.o_meta);
  for (int m = tid; m < n; m += NT) s_meta[m] = a.meta[(long long)c * n + m];
  for (int it = tid; it < ns * G; it += NT) {
    const int g = it / ns, i = it - g * ns;
    Cx<R> v(0, 0);
    if (g < gcount) v = cvt<R>(a.r[(long long)(g0 + g) * a.N + lo_c + i]);
    x[i * GS + g] = v;
  }
  __syncthreads();
  if (!L2X) cluster_sync();      // every CTA's mbarriers are ready before anyone arrives on them

  auto layer_of = [&](int s) { return s < n ? s : 2 * n - 2 - s; };
  auto last_col = [&](const uchar4& e) -> int { return dC == 0 ? 0 : dC == 1 ? e.x : dC == 2 ? e.y : dC == 3 ? e.z : e.w; };
  // first received slot of depth d: S_j columns-worth of partial sums for every depth j < d
  auto xbase = [&](const uchar4& e, int d) {
    int b = 0;
    if (d > 1) b += (int)e.x << (dC - 1);
    if (d > 2) b += ((int)e.y - e.x) << (dC - 2);
    if (d > 3) b += ((int)e.z - e.y) << (dC - 3);
    if (d > 4) b += ((int)e.w - e.z) << (dC - 4);
    return b;
  };
  const unsigned sm_u32 = smem_u32(sm);
  const unsigned bytesD = (unsigned)(ns * a.rsD * (int)sizeof(Cx<R>));
  auto record = [&](int s) { return a.pack + ((long long)layer_of(s) * C + c) * a.cap; };
  auto issue_D = [&](int s) {
    const int b = s & (a.dbufs - 1);
    fence_proxy_async();
    mbar_expect_tx(&barD[b], bytesD);
    bulk_g2s(sm + a.o_D[b], record(s), bytesD, &barD[b]);
  };
  auto issue_F = [&](int s, int W) {
    const unsigned bytes = (unsigned)(ns * slab_stride<R>(W) * (int)sizeof(Cx<R>));
    unsigned long long* mb = &barF[s & 1];
    if (bytes == 0) {
      mbar_arrive(mb);
    } else {
      fence_proxy_async();
      mbar_expect_tx(mb, bytes);
      bulk_g2s(sm + a.o_F[s & 1], record(s) + (long long)ns * a.rsD, bytes, mb);
    }
  };
  auto wait_copy = [&](unsigned long long* mb, unsigned parity, int m) {
    long long spins = 0;
    while (!mbar_try_wait(mb, parity))
      if (++spins > kWaitLimit) {
        report_error(a.status, HSWEEP_ERR_TIMEOUT, m);
        *s_fail = 1;
        break;
      }
  };

  // this thread's (row, right-hand side) of the update
  const int row0 = (warp * RG + lane / (CS * GL)) * RA;     // first row of this lane's group
  const int gl4 = (lane / CS) % GL;
  int urow, ug;
  bool uown;
  {
    Cx<R> dummy[RA * B];
#pragma unroll
    for (int j = 0; j < RA * B; ++j) dummy[j] = Cx<R>(0, 0);
    int idx;
    scatter_sum<R, RA * B, CS, 1>(dummy, lane, idx, uown);
    urow = row0 + idx / B;
    ug = gl4 * B + idx % B;
  }
  const bool ux = uown && urow < ns;
  uown = ux && ug < gcount;
  const long long upos = (long long)(g0 + ug) * a.N + lo_c + urow;
  // Its inputs come a step ahead by cp.async (registers loaded a step ahead were waited for at
  // once: 15 % of a step): r (forward) or w (backward) of every (row, right-hand side) by and for
  // its own thread, in one place, and the coupling of a row by its first lane
  const int slot = urow * G + ug;
  c128* in_r = reinterpret_cast<c128*>(sm + a.o_in) + slot;
  Cx<R>* in_w = reinterpret_cast<Cx<R>*>(in_r);
  Cx<R>* in_c = reinterpret_cast<Cx<R>*>(sm + a.o_inc) + urow;
  if (ux) *in_r = c128(0.0, 0.0);
  auto copy_in = [](Cx<R>* dst, const Cx<R>* src) {
    if constexpr (sizeof(R) == 4) cp_async8(dst, src);
    else cp_async16(dst, src);
  };
  auto load_inputs = [&](int s) {
    const bool fwd = s < n;
    const int m = layer_of(s);
    const int mn = (fwd && m < n - 1) ? m + 1 : m;
    if (ux && ug == 0) copy_in(in_c, a.cpl + (long long)mn * n + lo_c + urow);
    if (uown) {
      if (fwd) {
        if (m < n - 1) cp_async16(in_r, a.r + upos + (long long)(m + 1) * n);
      } else {
        copy_in(in_w, a.w + upos + (long long)m * n);
      }
    }
    cp_async_commit();
  };

  // the copies are issued by the last warp, which has the fewest column chunks
  const bool producer = tid == NT - 32;
  if (producer) {
    issue_F(0, last_col(s_meta[0]));
    issue_D(0);
  }
  int issuedF = 1, issuedD = 1;
  load_inputs(0);

  int t = 0;
  for (; t < nsteps; ++t) {
    const int par = t & 1;
    const unsigned ph = (unsigned)(t >> 1) & 1u;
    const int m = layer_of(t);
    const bool fwd = t < n;
    const uchar4 mc = s_meta[m];
    if (t + 1 < nsteps) {
      if (producer) {
        const int W1 = last_col(s_meta[layer_of(t + 1)]);
        issue_F(t + 1, W1);
        if (a.dbufs == 2) issue_D(t + 1);
        if (t + 2 < nsteps) {
          // the record after that into L2
          const int W2 = last_col(s_meta[layer_of(t + 2)]);
          const unsigned pb = bytesD + (unsigned)(ns * slab_stride<R>(W2) * (int)sizeof(Cx<R>));
          asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(record(t + 2)), "r"(pb) : "memory");
        }
      }
      issuedF = t + 2;
      if (a.dbufs == 2) issuedD = t + 2;
    }
    const int W = last_col(mc);
    const int rs = slab_stride<R>(W);
    const int nF = (W + KW - 1) / KW, nD = (ns + KW - 1) / KW;
    const Cx<R>* F = reinterpret_cast<const Cx<R>*>(sm + a.o_F[par]);
    const Cx<R>* D = reinterpret_cast<const Cx<R>*>(sm + a.o_D[t & (a.dbufs - 1)]);
    const int nFx = (a.Wcap + KW - 1) / KW;
    if (!L2X && C > 1 && tid == 0)
      mbar_expect_tx(&barX[par], (unsigned)(xbase(mc, dC + 1) * G * (int)sizeof(Cx<R>)));

    // column chunk of a matrix (row stride st, first column k0): out[k] = sum_i B[i][k] x[i]
    // for the columns below kend
    auto chunk = [&](const Cx<R>* mat, int st, int k0, auto put) {
      const int cl = lane % CL, gl = (lane / CL) % GL, rl = lane / (CL * GL);
      Cx<R> acc[A][B];
#pragma unroll
      for (int u = 0; u < A; ++u)
#pragma unroll
        for (int g = 0; g < B; ++g) acc[u][g] = Cx<R>(0, 0);
      const Cx<R>* bp = mat + rl * st + k0 + (A == 4 ? 2 * cl : cl);
      const Cx<R>* xp = x + rl * GS + gl * B;
#pragma unroll (G <= 2 ? 4 : 2)
      for (int i = rl; i < ns; i += RL, bp += RL * st, xp += RL * GS) {
        Cx<R> f[A];
        if constexpr (A == 4) {
          const float4 v0 = *reinterpret_cast<const float4*>(bp), v1 = *reinterpret_cast<const float4*>(bp + KW / 2);
          f[0] = Cx<R>(v0.x, v0.y);
          f[1] = Cx<R>(v0.z, v0.w);
          f[2] = Cx<R>(v1.x, v1.y);
          f[3] = Cx<R>(v1.z, v1.w);
        } else {
          f[0] = *bp;
        }
        Cx<R> xv[B];
        load_rhs(xp, xv);
#pragma unroll
        for (int u = 0; u < A; ++u) mac(acc[u], f[u], xv);
      }
      Cx<R> o[A * B];
#pragma unroll
      for (int u = 0; u < A; ++u)
#pragma unroll
        for (int g = 0; g < B; ++g) o[u * B + g] = acc[u][g];
      int idx;
      bool first;
      scatter_sum<R, A * B, RL, CL * GL>(o, lane, idx, first);
      constexpr int CNT = A * B / RL > 1 ? A * B / RL : 1;
      constexpr int PV = (VG == 2 && CNT >= 2 && B >= 2) ? 2 : 1;      // values per store
#pragma unroll
      for (int j = 0; j < CNT; j += PV) {
        const int u = (idx + j) / B, g = (idx + j) % B;
        const int k = k0 + (A == 4 ? 2 * cl + (u & 1) + (u >> 1) * (KW / 2) : cl);
        if (first) put(k, gl * B + g, o[j], o[j + PV - 1], std::integral_constant<int, PV>());
      }
    };

    // ---- 1. the ancestors' partial sums ------------------------------------------------
    wait_copy(&barF[par], ph, m);
    int ci = warp;
    if constexpr (L2X) {
      // every slot below Wcap is rewritten every step (zeros past the layer's columns), so
      // a slot holds this step's value or the one from two steps before, told apart by the tag
      typename T::W* dst = a.xch + (((long long)par * gridDim.x) + blockIdx.x) * a.Wcap * G;
      for (; ci < nFx; ci += NW) {
        chunk(F, rs, min(ci, nF - 1) * KW, [&](int kf, int g, Cx<R> v0, Cx<R> v1, auto pv) {
          static_assert(decltype(pv)::value == 2, "the L2 slots are written in pairs");
          const int k = kf + (ci - min(ci, nF - 1)) * KW;
          if (k < a.Wcap && (int)blockIdx.x != a.withhold) {
            const bool in = k < W;
            store_words(dst + k * G + g, T::pack(in ? v0 : Cx<R>(0, 0), ph), T::pack(in ? v1 : Cx<R>(0, 0), ph));
          }
        });
      }
    } else {
      for (; ci < nF; ci += NW)
        chunk(F, rs, ci * KW, [&](int k, int g, auto v0, auto v1, auto pv) {
          if (k < W && (int)blockIdx.x != a.withhold) {
            // column k of depth d: to the S CTAs of the sibling subtree, slot (c mod S, k)
            const int d = 1 + (k >= mc.x) + (dC > 1 && k >= mc.y) + (dC > 2 && k >= mc.z);
            const int S = 1 << (dC - d);
            const unsigned c0 = ((c >> (dC - d)) ^ 1) << (dC - d);
            const int e0 = d == 1 ? 0 : d == 2 ? mc.x : d == 3 ? mc.y : mc.z;
            const int e1 = d == 1 ? mc.x : d == 2 ? mc.y : d == 3 ? mc.z : mc.w;
            const int at = xbase(mc, d) + (c & (S - 1)) * (e1 - e0) + (k - e0);
            const unsigned off = (unsigned)(a.o_p[par] + (at * G + g) * (int)sizeof(Cx<R>));
            for (int u = 0; u < S; ++u) {
              const unsigned base = mapa(sm_u32, c0 + u);
              if constexpr (decltype(pv)::value == 2) send2(base + off, v0, v1, base + a.o_bar + 32 + 8 * par);
              else send(base + off, v0, base + a.o_bar + 32 + 8 * par);
            }
          }
        });
    }
    // ---- 2. the slab's own part, while the sums travel -----------------------------------
    if (a.dbufs == 2) wait_copy(&barD[par], ph, m);
    else wait_copy(&barD[0], (unsigned)t & 1u, m);
    for (; ci < (L2X ? nFx : nF) + nD; ci += NW)
      chunk(D, a.rsD, (ci - (L2X ? nFx : nF)) * KW, [&](int k, int g, Cx<R> v0, Cx<R> v1, auto pv) {
        if (k < ns) {
          yl[k * GS + g] = v0;
          if (decltype(pv)::value == 2) yl[k * GS + g + 1] = v1;
        }
      });
    // ---- 3. the sums over the sibling subtrees ------------------------------------------
    if (C > 1) {
      constexpr int IPC = G / VG;      // words per column
      const int items = W * IPC;
      if constexpr (!L2X) {
        if (tid < items) {
          long long spins = 0;
          while (!mbar_try_wait(&barX[par], ph)) {
            ++spins;
            if (spins > a.wait_limit || ((spins & 63) == 0 && *(volatile int*)a.status != 0)) {
              report_error(a.status, HSWEEP_ERR_TIMEOUT, m);
              *s_fail = 1;
              break;
            }
          }
        }
      }
      for (int it = tid; it < items; it += NT) {
        const int k = it / IPC, gv = (it - k * IPC) * VG;
        const int d = 1 + (k >= mc.x) + (dC > 1 && k >= mc.y) + (dC > 2 && k >= mc.z);
        const int S = 1 << (dC - d);
        Cx<R> v[8][VG];
        if constexpr (!L2X) {
          const int e0 = d == 1 ? 0 : d == 2 ? mc.x : d == 3 ? mc.y : mc.z;
          const int e1 = d == 1 ? mc.x : d == 2 ? mc.y : d == 3 ? mc.z : mc.w;
          const Cx<R>* src = reinterpret_cast<const Cx<R>*>(sm + a.o_p[par]) + (xbase(mc, d) + (k - e0)) * G + gv;
          const int us = (e1 - e0) * G;
#pragma unroll
          for (int u = 0; u < 8; ++u)
            if (u < S) {
              if constexpr (VG == 2) {
                const float4 w4 = *reinterpret_cast<const float4*>(src + u * us);
                v[u][0] = Cx<R>(w4.x, w4.y);
                v[u][1] = Cx<R>(w4.z, w4.w);
              } else {
                v[u][0] = src[u * us];
              }
            }
        } else {
          const int c0 = ((c >> (dC - d)) ^ 1) << (dC - d);
          const long long cs = (long long)a.Wcap * G;
          const typename T::W* src = a.xch + ((long long)par * gridDim.x + (blockIdx.x - c) + c0) * cs + k * G + gv;
          typename T::W wv[8][VG];
#pragma unroll
          for (int u = 0; u < 8; ++u)
            if (u < S) load_words(src + u * cs, wv[u]);
          long long spins = 0;
          for (;;) {      // re-read every word not yet written for this step
            bool pending = false;
#pragma unroll
            for (int u = 0; u < 8; ++u)
              if (u < S && !(T::ok(wv[u][0], ph) && T::ok(wv[u][VG - 1], ph))) {
                load_words(src + u * cs, wv[u]);
                pending = true;
              }
            if (!pending) break;
            if (++spins > a.wait_limit || ((spins & 63) == 0 && *(volatile int*)a.status != 0)) {
              report_error(a.status, HSWEEP_ERR_TIMEOUT, m);
              *s_fail = 1;
              break;
            }
          }
#pragma unroll
          for (int u = 0; u < 8; ++u)
            if (u < S)
#pragma unroll
              for (int j = 0; j < VG; ++j) v[u][j] = T::value(wv[u][j]);
        }
        // pairwise: a short chain (the additions of FP64 are slow)
#pragma unroll
        for (int o = 1; o < 8; o <<= 1)
          if (o < S)
#pragma unroll
            for (int u = 0; u + o < 8; u += 2 * o)
              if (u + o < S)
#pragma unroll
                for (int j = 0; j < VG; ++j) v[u][j] += v[u + o][j];
        if constexpr (VG == 2) *reinterpret_cast<float4*>(q + k * GS + gv) = make_float4(v[0][0].re, v[0][0].im, v[0][1].re, v[0][1].im);
        else q[k * GS + gv] = v[0][0];
      }
    }
    __syncthreads();
    if (*s_fail != 0) break;
    if (a.dbufs == 1 && t + 1 < nsteps) {
      if (producer) issue_D(t + 1);
      issuedD = t + 2;
    }
    // ---- 4. y = D x + F q and the update --------------------------------------------------
    {
      if (warp * RG * RA < ns) {
      const int cs = lane % CS;
      Cx<R> acc[RA][B];
#pragma unroll
      for (int u = 0; u < RA; ++u)
#pragma unroll
        for (int g = 0; g < B; ++g) acc[u][g] = Cx<R>(0, 0);
      {
        const Cx<R>* Fr[RA];
#pragma unroll
        for (int u = 0; u < RA; ++u) Fr[u] = F + min(row0 + u, ns - 1) * rs;
#pragma unroll (G <= 2 ? 4 : 2)
        for (int k = cs; k < W; k += CS) {
          Cx<R> f[RA];
#pragma unroll
          for (int u = 0; u < RA; ++u) f[u] = Fr[u][k];
          Cx<R> v[B];
          load_rhs(q + k * GS + gl4 * B, v);
#pragma unroll
          for (int u = 0; u < RA; ++u) mac(acc[u], f[u], v);
        }
      }
      Cx<R> o[RA * B];
#pragma unroll
      for (int u = 0; u < RA; ++u)
#pragma unroll
        for (int g = 0; g < B; ++g) o[u * B + g] = acc[u][g];
      int idx;
      bool first;
      scatter_sum<R, RA * B, CS, 1>(o, lane, idx, first);
      cp_async_wait0();
      __syncwarp();
      if (ux) {
        const Cx<R> y = o[0] + yl[urow * GS + ug];
        const Cx<R> cpl = *in_c;
        const long long pos = upos + (long long)m * n;
        Cx<R> xn;
        if (fwd) {
          if (m < n - 1) {
            if (uown) a.w[pos] = y;
            xn = cvt<R>(*in_r) - cpl * y;
          } else {
            if (uown) a.z[pos] = cvt<double>(y);
            xn = cpl * y;
          }
        } else {
          const Cx<R> uu = uown ? *in_w - y : Cx<R>(0, 0);
          if (uown) a.z[pos] = cvt<double>(uu);
          xn = cpl * uu;
        }
        x[urow * GS + ug] = xn;
      }
      }
      __syncwarp();       // a row's lanes have read its coupling: its first lane may replace it
      if (t + 1 < nsteps) load_inputs(t + 1);
    }
    __syncthreads();
  }
  // a CTA that stopped early still owns the copies it issued: wait for them
  cp_async_wait0();
  if (producer && t < nsteps) {
    for (int s = t; s < issuedF; ++s) {
      long long spins = 0;
      while (!mbar_try_wait(&barF[s & 1], (unsigned)(s >> 1) & 1u) && ++spins <= kWaitLimit) {
      }
    }
    for (int s = t; s < issuedD; ++s) {
      long long spins = 0;
      unsigned long long* mb = a.dbufs == 2 ? &barD[s & 1] : &barD[0];
      const unsigned pp = a.dbufs == 2 ? (unsigned)(s >> 1) & 1u : (unsigned)s & 1u;
      while (!mbar_try_wait(mb, pp) && ++spins <= kWaitLimit) {
      }
    }
  }
  __syncthreads();
  if (!L2X) cluster_sync();      // no CTA leaves while another may still read its shared memory
}

// ---- packing: the slab records of layers m0 .. from the factor store ---------------------------
// One CTA per (slab, layer), or eight when one layer is packed at a time.  D^t[j][i] = T(i, j): the leaf block, or the product of the
// factors of the two children that part rows i and j (rank(v) terms).
template <typename R>
__global__ void __launch_bounds__(256) pack_slabs(int m0, int L, int leaf, int nnodes, int dC, int rsD,
                                                  const int* __restrict__ lo, const int* __restrict__ sz,
                                                  const long long* __restrict__ off, const Cx<R>* __restrict__ leaves,
                                                  const Cx<R>* __restrict__ fac, long long layer_stride,
                                                  const int* __restrict__ rank,
                                                  Cx<R>* __restrict__ pack, long long cap, int n, uchar4* __restrict__ meta) {
  const int c = blockIdx.x, C = 1 << dC, m = m0 + blockIdx.y;
  const int vc = C + c, lo_c = lo[vc], ns = sz[vc];
  const int t0 = blockIdx.z * blockDim.x + threadIdx.x, nt = gridDim.z * blockDim.x;
  // layer_stride = 0: a single layer (the setup's buffers), ranks and factors at their start
  const int* rk = layer_stride ? rank + (long long)m * nnodes : rank;
  const Cx<R>* F = fac + (long long)m * layer_stride;
  const Cx<R>* D = leaves + (long long)m * layer_stride;
  Cx<R>* out = pack + ((long long)m * C + c) * cap;
  int e[4] = {0, 0, 0, 0}, W = 0;
  for (int d = 1; d <= dC; ++d) {
    W += max(1, rk[vc >> (dC - d)]);
    e[d - 1] = W;
  }
  if (t0 == 0) meta[(long long)c * n + m] = make_uchar4(e[0], e[1], e[2], e[3]);
  auto leaf_of = [&](int i) {
    int v = vc;
    for (int d = dC; d < L; ++d) v = 2 * v + ((lo_c + i) >= lo[2 * v + 1] ? 1 : 0);
    return v;
  };
  for (int it = t0; it < ns * rsD; it += nt) {
    const int j = it / rsD, i = it - j * rsD;
    Cx<R> val(0, 0);
    if (i < ns) {
      int vi = leaf_of(i), vj = leaf_of(j);
      if (vi == vj) {
        val = D[(long long)(vi - (1 << L)) * leaf * leaf + (long long)(lo_c + j - lo[vj]) * leaf + (lo_c + i - lo[vi])];
      } else {
        while ((vi >> 1) != (vj >> 1)) { vi >>= 1; vj >>= 1; }
        const Cx<R>* Fi = F + off[vi] + (lo_c + i - lo[vi]);
        const Cx<R>* Fj = F + off[vj] + (lo_c + j - lo[vj]);
        const int r = rk[vi], si = sz[vi], sj = sz[vj];
        for (int k = 0; k < r; ++k) cfma(val, Fi[(long long)k * si], Fj[(long long)k * sj]);
      }
    }
    out[it] = val;
  }
  const int rs = slab_stride<R>(W);
  Cx<R>* fo = out + (long long)ns * rsD;
  for (int it = t0; it < ns * rs; it += nt) {
    const int i = it / rs, k = it - i * rs;
    Cx<R> val(0, 0);
    if (k < W) {
      const int d = 1 + (k >= e[0]) + (dC > 1 && k >= e[1]) + (dC > 2 && k >= e[2]);
      const int v = vc >> (dC - d);
      const int kk = k - (d == 1 ? 0 : e[d - 2]);
      if (kk < rk[v]) val = F[off[v] + (long long)kk * sz[v] + (lo_c + i - lo[v])];
    }
    fo[it] = val;
  }
}

__global__ void narrow_couplings(const c128* __restrict__ in, c64* __restrict__ out, long long cnt) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < cnt; i += (long long)gridDim.x * blockDim.x)
    out[i] = cvt<float>(in[i]);
}

static long long al(long long x, long long b) { return (x + b - 1) / b * b; }

struct SlabConfig {
  bool ok = false, l2x = false;
  int G = 0, dbufs = 0, groups = 0, per_launch = 0;   // groups of G right-hand sides; of them one launch runs
  size_t smem = 0;
  long long cost = 0;                                 // estimated ns a step of the batch
};

// shared-memory plan for G right-hand sides; returns total bytes
template <typename R>
static size_t slab_plan(const hsweep_s* h, int G, int dbufs, bool l2x, SlabArgs<R>& a) {
  const size_t es = sizeof(Cx<R>);
  const int nsm = h->tree.maxsz(h->slab_dC), GS = vstride<R>(G);
  const int Wp = slab_stride<R>(h->slab_W);
  size_t o = 0;
  for (int b = 0; b < 2; ++b) { a.o_F[b] = (unsigned)o; o += al(((long long)nsm * Wp + (Wp ? kKW : 0)) * es, 128); }
  for (int b = 0; b < 2; ++b) {
    if (b < dbufs) { a.o_D[b] = (unsigned)o; o += al(((long long)nsm * h->slab_rsD + kKW) * es, 128); }
    else a.o_D[b] = a.o_D[0];
  }
  a.o_x = (unsigned)o; o += al((long long)nsm * GS * es, 16);
  a.o_q = (unsigned)o; o += al((long long)std::max(1, h->slab_W) * GS * es, 16);
  for (int b = 0; b < 2; ++b) { a.o_p[b] = (unsigned)o; o += l2x ? 0 : al((long long)h->slab_X * G * es, 16); }
  a.o_y = (unsigned)o; o += al((long long)nsm * GS * es, 16);
  a.o_in = (unsigned)o; o += (size_t)nsm * G * sizeof(c128);
  a.o_inc = (unsigned)o; o += al((long long)nsm * es, 16);
  a.o_bar = (unsigned)o; o += 64;
  a.o_meta = (unsigned)o; o += al((long long)h->n * sizeof(uchar4), 16);
  a.dC = h->slab_dC;
  a.C = 1 << h->slab_dC;
  a.rsD = h->slab_rsD;
  a.dbufs = dbufs;
  a.Wcap = h->slab_W;
  return o;
}

template <typename R> using SlabKernel = void (*)(SlabArgs<R>);

// Threads per CTA: a step of one or two right-hand sides is a few hundred instructions a
// warp, most of them overhead that every further warp repeats; with four on a slab of at most
// 32 rows, two CTAs of 256 threads share an SM and cover each other's waits (n = 511, 64
// right-hand sides: 4.5 us a step against 4.7 with eight in one CTA).
constexpr int slab_threads(int G, int rows, bool fp64) { return fp64 || G <= 2 || (G == 4 && rows <= 32) ? 256 : 512; }

template <typename R, int G, bool L2X>
static SlabKernel<R> slab_kernel_g(int rows) {
  if constexpr (sizeof(R) == 4) {
    // step 4: a warp per group of RA rows, every lane a column slice; all warps busy
    constexpr int CS = 32 / (G / Tile<float, G>::B);
    constexpr int NT = slab_threads(G, 32, false), NT64 = slab_threads(G, 64, false);
    if (rows <= 16) return sweep_slab_kernel<float, G, 512 / NT, CS, NT, L2X>;
    if (rows <= 32) return sweep_slab_kernel<float, G, 2 * 512 / NT, CS, NT, L2X>;
    return sweep_slab_kernel<float, G, 4 * 512 / NT64, CS, NT64, L2X>;
  } else {
    // eight warps, two a sub-core, whatever the slab: the FP64 unit is the bound, and fewer
    // lanes a row mean fewer additions to join them
    if (rows <= 8) return sweep_slab_kernel<double, G, 1, 16, 256, L2X>;
    if (rows <= 16) return sweep_slab_kernel<double, G, 1, 8, 256, L2X>;
    return sweep_slab_kernel<double, G, 1, 4, 256, L2X>;
  }
}
template <typename R>
static SlabKernel<R> slab_kernel(int G, int rows, bool l2x) {
  if constexpr (sizeof(R) == 4)
    if (l2x) return G == 8 ? slab_kernel_g<R, 8, true>(rows) : slab_kernel_g<R, 4, true>(rows);
  switch (G) {
    case 1: return slab_kernel_g<R, 1, false>(rows);
    case 2: return slab_kernel_g<R, 2, false>(rows);
  }
  if constexpr (sizeof(R) == 4) return G == 4 ? slab_kernel_g<R, 4, false>(rows) : slab_kernel_g<R, 8, false>(rows);
  return nullptr;
}

template <typename R>
static bool launch_config(const hsweep_s* h, SlabKernel<R> kern, const SlabConfig& c, int groups, cudaLaunchConfig_t& lc,
                          cudaLaunchAttribute* at) {
  const int C = 1 << h->slab_dC;
  if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)c.smem) != cudaSuccess ||
      (!c.l2x && C > 8 && cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess)) {
    cudaGetLastError();
    return false;
  }
  lc = cudaLaunchConfig_t{};
  lc.blockDim = dim3(slab_threads(c.G, h->tree.maxsz(h->slab_dC), sizeof(R) == 8));
  lc.gridDim = dim3(C * groups);
  lc.dynamicSmemBytes = c.smem;
  lc.stream = h->stream;
  if (c.l2x) {
    at[0].id = cudaLaunchAttributeCooperative;
    at[0].val.cooperative = 1;
  } else {
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = C;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
  }
  lc.attrs = at;
  lc.numAttrs = 1;
  return true;
}

template <typename R>
static SlabConfig choose_slab_uncached(const hsweep_s* h, int nrhs) {
  SlabConfig best;
  if (!h->slab_valid) return best;
  const int C = 1 << h->slab_dC, rows = h->tree.maxsz(h->slab_dC);
  double best_cost = 1e300;
  struct Try { bool l2x; int G; };
  const Try tries[] = {{false, 8}, {false, 4}, {false, 2}, {false, 1}, {true, 8}, {true, 4}};
  for (const Try& y : tries) {
    // complex128 is bound by the FP64 units, which the team sweep's smaller teams load
    // better once a cluster would carry more than two right-hand sides (n = 255, 16 of
    // them: 12.7 against 10.8 us a step)
    if (sizeof(R) == 8 && (y.G > 2 || y.l2x)) continue;
    if (y.l2x && C == 1) continue;
    for (int dbufs : {2, 1}) {
      SlabArgs<R> a;
      SlabConfig c;
      c.l2x = y.l2x;
      c.G = y.G;
      c.dbufs = dbufs;
      c.smem = slab_plan<R>(h, c.G, dbufs, c.l2x, a);
      if (c.smem > 227 * 1024) continue;
      cudaLaunchConfig_t lc;
      cudaLaunchAttribute at[1];
      SlabKernel<R> kern = slab_kernel<R>(c.G, rows, c.l2x);
      if (!launch_config<R>(h, kern, c, 1, lc, at)) continue;
      int act = 0, per_sm = 0;     // teams that run at a time
      if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, (int)lc.blockDim.x, c.smem) != cudaSuccess) {
        cudaGetLastError();
        continue;
      }
      if (c.l2x) {
        act = per_sm * h->num_sms / C;
      } else if (cudaOccupancyMaxActiveClusters(&act, kern, &lc) != cudaSuccess) {
        cudaGetLastError();
        continue;
      }
      if (act < 1) continue;
      c.groups = (nrhs + c.G - 1) / c.G;
      c.per_launch = c.l2x ? std::min(c.groups, act) : c.groups;
      const int rounds = (c.groups + act - 1) / act;
      if (sizeof(R) == 8 && rounds > 1) continue;
      // Microseconds a step (complex64, fitted to n = 127, 300, 511, 700 and 1023 with 1 to 64
      // right-hand sides): a latency, 0.35 more for an exchange through L2, and work per
      // right-hand side that two CTAs on an SM share it for (clusters double up as soon as
      // there are more than fit with an SM each)
      const double rc = rows * (2.0 * h->slab_W + rows);
      const int alone = c.l2x ? h->num_sms / C : std::max(1, act / per_sm);
      const int shared = (std::min(c.groups, act) + alone - 1) / alone;
      const double work = (0.12 + 1.8e-5 * rc) * c.G * (sizeof(R) == 4 ? 1.0 : 15.0);
      const double cost = rounds * (1.75 + 2.5e-5 * rc + (c.l2x ? 0.35 : 0.0) + shared * work);
      if (cost < best_cost - 1e-9) {
        best_cost = cost;
        best = c;
        best.ok = true;
        best.cost = (long long)(1e3 * cost);
      }
      break;      // two D stages where they fit
    }
  }
  return best;
}

// complex128 with two right-hand sides a cluster against the team sweep, by estimates fitted to
// n = 130 to 511, ranks 16 to 56 at the top and 8 to 14 right-hand sides.  Microseconds a step
// (slabs, teams): n = 255, 8 RHS 7.1, 8.2, 10 RHS 7.1, 10.3; n = 300, 8 RHS 9.5, 9.4, 10 RHS 9.5, 12.7;
// n = 511, 8 RHS 14.8, 12.3, 10 RHS 14.8, 20.7 (eps_H = 1e-6); the slabs' lead falls with the rank
// (n = 257, top rank 46: 8 RHS 17.4, 11.3; 10 RHS 17.4, 16.4), so beyond 16 rows a slab has to be
// ahead by 15 %.  One a cluster was never the slower (n = 64 to 511: 0.50 to 0.98 of the teams' time).
static bool slower_than_teams(hsweep_s* h, int nrhs) {
  const double other = 1e-3 * (double)hsw_team_cost(h, nrhs);
  if (other <= 0) return false;
  const int rows = h->tree.maxsz(h->slab_dC);
  const double W = h->slab_W, rc = rows * (2.0 * W + rows);
  return rows <= 16 ? 2.5 + 0.028 * W + 1.72e-3 * rc > 1.1 * other : 1.15 * (3.65 + 0.0563 * W + 1.24e-3 * rc) > other;
}

template <typename R>
static SlabConfig choose_slab(hsweep_s* h, int nrhs) {
  for (const auto& e : h->slab_plans)
    if (e[0] == nrhs) {
      SlabConfig s;
      s.ok = e[1] != 0; s.l2x = e[2] != 0; s.G = (int)e[3]; s.dbufs = (int)e[4]; s.groups = (int)e[5];
      s.per_launch = (int)e[6]; s.smem = (size_t)e[7]; s.cost = e[8];
      return s;
    }
  SlabConfig s = choose_slab_uncached<R>(h, nrhs);
  if (sizeof(R) == 8 && s.ok && s.G == 2 && slower_than_teams(h, nrhs)) s.ok = false;
  if (h->slab_plans.size() >= 64) h->slab_plans.erase(h->slab_plans.begin());
  h->slab_plans.push_back({nrhs, s.ok ? 1 : 0, s.l2x ? 1 : 0, s.G, s.dbufs, s.groups, s.per_launch, (long long)s.smem,
                           s.cost});
  return s;
}

template <typename R>
static int apply_slab_impl(hsweep_s* h, const c128* r, c128* z, int nrhs, bool* used, void* scratch, size_t scratch_bytes) {
  const SlabConfig cfg = choose_slab<R>(h, nrhs);
  if (!cfg.ok) return HSWEEP_OK;
  const long long es = sizeof(Cx<R>);
  const int C = 1 << h->slab_dC;
  const long long wb = al((long long)nrhs * h->N * es, 256);
  const long long xb = cfg.l2x ? 2LL * cfg.per_launch * C * h->slab_W * cfg.G * es : 0;
  void* wptr = scratch;
  void* xptr = h->noalloc_slots;
  if (scratch) {      // the scratch of hsweep_apply_noalloc, and its array for the exchange slots
    if (wb > (long long)scratch_bytes || xb > (long long)h->noalloc_slot_bytes) return HSWEEP_OK;
  } else {
    const long long need_w = (long long)nrhs * h->N;
    if (need_w > h->wcache_cap) {
      int rc = hsw_regrow(h, &h->d_wcache, (size_t)(need_w * es));
      if (rc) {
        if (!h->d_wcache) h->wcache_cap = 0;
        return rc;
      }
      h->wcache_cap = need_w;
    }
    // room for the largest exchange of any plan for as many right-hand sides or fewer,
    // although this call may need none: a captured call with fewer of them can have a plan
    // that exchanges through L2, and must not allocate
    // (in complex128 the team sweep serves some counts between those of the slabs)
    const long long xcap = std::max({hsw_slab_exchange_bound(h), hsw_strong_exchange_bound(h, nrhs),
                                     sizeof(R) == 8 ? hsw_team_exchange_bound(h, nrhs) : 0LL});
    const long long need_x = std::max(xb, xcap) / es;
    if (need_x > h->xch_cap) {
      int rc = hsw_regrow(h, &h->d_xch, (size_t)(need_x * es));
      if (rc) {
        if (!h->d_xch) h->xch_cap = 0;
        return rc;
      }
      h->xch_cap = need_x;
    }
    wptr = h->d_wcache;
    xptr = h->d_xch;
  }
  SlabArgs<R> a;
  slab_plan<R>(h, cfg.G, cfg.dbufs, cfg.l2x, a);
  a.n = h->n; a.nrhs = nrhs; a.N = h->N; a.cap = h->slab_cap;
  a.lo = h->d_lo; a.sz = h->d_sz; a.meta = reinterpret_cast<const uchar4*>(h->d_slab_meta);
  a.pack = reinterpret_cast<const Cx<R>*>(h->d_slab);
  a.cpl = reinterpret_cast<const Cx<R>*>(h->d_slab_cpl ? h->d_slab_cpl : h->d_north_m); a.r = r; a.z = z;
  a.w = reinterpret_cast<Cx<R>*>(wptr);
  a.xch = reinterpret_cast<typename Tagged<R>::W*>(xptr);
  a.status = h->d_status;
  // test hooks (environment), as in sweep_team.cu
  a.wait_limit = kWaitLimit;
  a.withhold = -1;
  if (const char* e = getenv("HSWEEP_TEST_WAIT_LIMIT")) {
    const long long v = atoll(e);
    if (v > 0 && v < kWaitLimit) a.wait_limit = v;
  }
  if (const char* e = getenv("HSWEEP_TEST_WITHHOLD")) a.withhold = atoi(e);
  SlabKernel<R> kern = slab_kernel<R>(cfg.G, h->tree.maxsz(h->slab_dC), cfg.l2x);
  const bool prof = h->prof && !scratch;    // the no-allocation path creates no events
  cudaEvent_t e0 = nullptr, e1 = nullptr;
  if (prof) {
    for (cudaEvent_t* e : {&e0, &e1}) {
      if (!h->ev_free.empty()) { *e = h->ev_free.back(); h->ev_free.pop_back(); }
      else HSW_CUDA(cudaEventCreate(e));
    }
    HSW_CUDA(cudaEventRecord(e0, h->stream));
  }
  for (a.group0 = 0; a.group0 < cfg.groups; a.group0 += cfg.per_launch) {
    const int groups = std::min(cfg.per_launch, cfg.groups - a.group0);
    cudaLaunchConfig_t lc;
    cudaLaunchAttribute at[1];
    if (!launch_config<R>(h, kern, cfg, groups, lc, at)) return HSWEEP_ERR_CUDA;
    // every exchange slot starts with the tag bit set: steps 0 and 1 expect it clear
    if (cfg.l2x) HSW_CUDA(cudaMemsetAsync(xptr, 0xff, (size_t)xb, h->stream));
    HSW_CUDA(cudaLaunchKernelEx(&lc, kern, a));
    h->nlaunch += 1;
  }
  if (prof) {
    HSW_CUDA(cudaEventRecord(e1, h->stream));
    h->ev_sweep.push_back({e0, e1});
  }
  *used = true;
  return HSWEEP_OK;
}

}  // namespace

// The slab sweep serves the automatic plan: sweep_kernel 1 or 2, an explicit team, group or
// thread choice, and the tensor-core option, ask for other sweeps; the strongly admissible
// format in complex128 runs on its records.  Such a handle reserves and packs no slabs (at
// n = 1023 in complex64 they are 2.2 GB).
static bool slab_wanted(const hsweep_s* h) {
  const hsweep_opts& o = h->opt;
  return o.sweep_kernel == 0 && o.team == 0 && o.groups == 0 && o.team_threads == 0 && o.sweep_tc == 0 &&
         !(h->strong_R > 0 && h->prec == HSWEEP_FP64);
}

// The slab geometry: clusters of at most 16 CTAs (the largest that sm_103 schedules) and at
// most 64 rows per slab in complex64, 32 in complex128.
int hsw_slab_create(hsweep_s* h) {
  if (!slab_wanted(h)) return HSWEEP_OK;
  const size_t es = h->fac_elem();
  const int cap_rows = h->prec == HSWEEP_FP64 ? 32 : 64;
  int target = h->prec == HSWEEP_FP64 ? 16 : 32;
  int dC = 0;
  while (dC < 4 && dC < h->L && h->tree.maxsz(dC) > target) ++dC;
  if (h->tree.maxsz(dC) > cap_rows) return HSWEEP_OK;       // too large: the team sweep
  h->slab_dC = dC;
  const int nsm = h->tree.maxsz(dC);
  const bool f32 = es == sizeof(c64);
  h->slab_rsD = f32 ? slab_stride<float>(nsm) : slab_stride<double>(nsm);
  const int wmax = dC * h->r_max;
  h->slab_cap = al((long long)nsm * (h->slab_rsD + (f32 ? slab_stride<float>(wmax) : slab_stride<double>(wmax))), 16);
  int rc = HSWEEP_OK;
  if (f32) {
    const long long cnt = (long long)(h->n + 1) * h->n;
    if ((rc = hsw_alloc(h, &h->d_slab_cpl, (size_t)cnt * sizeof(c64)))) return rc;
    narrow_couplings<<<304, 256, 0, h->stream>>>(h->d_north_m, static_cast<c64*>(h->d_slab_cpl), cnt);
    h->nlaunch += 1;
    HSW_CUDA(cudaGetLastError());
  }
  rc = hsw_alloc(h, &h->d_slab, (size_t)h->n * (1 << dC) * h->slab_cap * es);
  if (rc) return rc;
  return hsw_alloc(h, &h->d_slab_meta, (size_t)h->n * (1 << dC) * sizeof(uchar4));
}

int hsw_pack_slabs(hsweep_s* h, int m0, int m1, const std::vector<int>& rk) {
  if (!h->d_slab || m1 <= m0) return HSWEEP_OK;
  if (h->slab_strong) {
    if (h->spack_valid) return HSWEEP_OK;     // the setup wrote them (hsw_strong_slabs)
    h->slab_strong = false;                   // a layer was replaced: all of them from the store
    m0 = 0;
    m1 = h->n;
  }
  const dim3 grid(1 << h->slab_dC, m1 - m0);
  if (h->prec == HSWEEP_FP64)
    pack_slabs<double><<<grid, 256, 0, h->stream>>>(m0, h->L, h->leaf, h->nnodes, h->slab_dC, h->slab_rsD, h->d_lo, h->d_sz,
        h->d_off, (const c128*)h->d_fac, (const c128*)h->d_fac, h->layer_stride, h->d_rank, (c128*)h->d_slab, h->slab_cap, h->n, (uchar4*)h->d_slab_meta);
  else
    pack_slabs<float><<<grid, 256, 0, h->stream>>>(m0, h->L, h->leaf, h->nnodes, h->slab_dC, h->slab_rsD, h->d_lo, h->d_sz,
        h->d_off, (const c64*)h->d_fac, (const c64*)h->d_fac, h->layer_stride, h->d_rank, (c64*)h->d_slab, h->slab_cap, h->n, (uchar4*)h->d_slab_meta);
  h->nlaunch += 1;
  HSW_CUDA(cudaGetLastError());
  // the setup and the import return with the work done: another stream may be set next
  HSW_CUDA(cudaStreamSynchronize(h->stream));
  // the most columns of any layer and slab, for the shared-memory plan
  const int dC = h->slab_dC, C = 1 << dC;
  h->slab_W = h->slab_X = 0;
  for (int m = 0; m < h->n; ++m)
    for (int c = 0; c < C; ++c) {
      int W = 0, X = 0;
      for (int d = 1; d <= dC; ++d) {
        const int r = std::max(1, rk[(size_t)m * h->nnodes + ((C + c) >> (dC - d))]);
        W += r;
        X += r << (dC - d);
      }
      h->slab_W = std::max(h->slab_W, W);
      h->slab_X = std::max(h->slab_X, X);
    }
  h->slab_plans.clear();
  h->slab_valid = true;
  return HSWEEP_OK;
}

// The strongly admissible T~_m as slabs, from the expanded factors of the setup (sibling-pair
// factors of rank 3R(L - l) + one leaf at depth l, zero outside each column's own cluster).
// The sweep on them does more arithmetic than the one on the records of sweep_strong.cu, which
// skips those zeros, but has one exchange and fewer barriers a step where that one gathers
// every cluster's interaction list.  Microseconds a step, complex64, R = 2 (records, slabs):
// n = 255, 1 RHS 2.95, 1.96; n = 511, 1 RHS 3.21, 2.47; 8 RHS 3.50, 2.81; 16 RHS 3.50, 3.54;
// 24 RHS 3.87, 3.55; 64 RHS 4.69, 5.62; n = 1023, 1 RHS 3.67, 2.99; 64 RHS 7.07, 9.07.
// complex128 keeps the records: the FP64 units pay for the zeros (n = 127, 1 RHS 5.02, 5.68;
// n = 511 7.86, 13.66).
int hsw_strong_slabs(hsweep_s* h, int m, const void* G_F, const void* G_leaf, const long long* d_gfo, const int* G_rank) {
  if (!h->d_slab || h->L < 2) return HSWEEP_OK;
  pack_slabs<float><<<dim3(1 << h->slab_dC, 1, 8), 256, 0, h->stream>>>(m, h->L, h->leaf, h->nnodes, h->slab_dC,
      h->slab_rsD, h->d_lo, h->d_sz, d_gfo, (const c64*)G_leaf, (const c64*)G_F, 0, G_rank, (c64*)h->d_slab,
      h->slab_cap, h->n, (uchar4*)h->d_slab_meta);
  h->nlaunch += 1;
  HSW_CUDA(cudaGetLastError());
  if (m < h->n - 1) return HSWEEP_OK;
  const int dC = h->slab_dC, C = 1 << dC;
  h->slab_W = h->slab_X = 0;
  for (int c = 0; c < C; ++c) {
    int W = 0, X = 0;
    for (int d = 1; d <= dC; ++d) {
      int b = ((C + c) >> (dC - d)) | 1;                    // the pair's right child, and its first leaf
      while (b < h->nleaves) b *= 2;
      const int r = 3 * h->strong_R * (h->L - d) + h->tree.sz[b];
      W += r;
      X += r << (dC - d);
    }
    h->slab_W = std::max(h->slab_W, W);
    h->slab_X = std::max(h->slab_X, X);
  }
  h->slab_plans.clear();
  h->slab_strong = h->slab_valid = true;
  return HSWEEP_OK;
}

// The faster of the two sweeps on the strongly admissible format, by the estimates that chose
// their plans (over n = 63 to 1023 and 1 to 64 RHS it misses the faster one only where the two
// are within 8 %)
int hsw_strong_prefers_slabs(hsweep_s* h, int nrhs) {
  if (!h->slab_strong || !h->spack_valid) return 0;
  const SlabConfig s = choose_slab<float>(h, nrhs);
  const long long other = s.ok ? hsw_strong_cost(h, nrhs) : 0;
  return s.ok && (other == 0 || s.cost < other);
}

// two CTAs on every SM, eight right-hand sides a team
long long hsw_slab_exchange_bound(const hsweep_s* h) {
  if (!h->slab_valid || h->prec == HSWEEP_FP64 || h->slab_dC == 0) return 0;
  return 2LL * 2 * h->num_sms * h->slab_W * 8 * (long long)h->fac_elem();
}

int hsw_slab_plan(hsweep_s* h, int nrhs, long long* out) {
  const SlabConfig s = h->prec == HSWEEP_FP64 ? choose_slab<double>(h, nrhs) : choose_slab<float>(h, nrhs);
  if (!s.ok) return 0;
  const int rows = h->tree.maxsz(h->slab_dC);
  const int st = h->prec == HSWEEP_FP64 ? slab_stride<double>(h->slab_W) : slab_stride<float>(h->slab_W);
  out[0] = h->slab_strong ? 3 : 2; out[1] = 1 << h->slab_dC; out[2] = s.G; out[3] = s.per_launch; out[4] = slab_threads(s.G, h->tree.maxsz(h->slab_dC), h->prec == HSWEEP_FP64);
  out[5] = (long long)s.smem; out[6] = (long long)rows * (st + h->slab_rsD) * (long long)h->fac_elem(); out[7] = s.l2x ? 1 : 0;
  return 1;
}

int hsw_apply_slab(hsweep_s* h, const c128* r, c128* z, int nrhs, bool* used, void* scratch, size_t scratch_bytes) {
  *used = false;
  if (h->prec == HSWEEP_FP64) return apply_slab_impl<double>(h, r, z, nrhs, used, scratch, scratch_bytes);
  return apply_slab_impl<float>(h, r, z, nrhs, used, scratch, scratch_bytes);
}
