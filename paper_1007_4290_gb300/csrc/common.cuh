// Shared device helpers: complex arithmetic templated on the real type, launch
// checks, and the status word every kernel reports device-side failures through.
#pragma once
#include <cuda_runtime.h>
#include <cstdint>
#include <cmath>

#include "../../include/hsweep.h"

template <typename R>
struct alignas(2 * sizeof(R)) Cx {
  R re, im;
  Cx() = default;
  __host__ __device__ constexpr Cx(R a, R b = R(0)) : re(a), im(b) {}
};

using c64 = Cx<float>;
using c128 = Cx<double>;

template <typename R> __host__ __device__ __forceinline__ Cx<R> operator+(Cx<R> a, Cx<R> b) { return Cx<R>(a.re + b.re, a.im + b.im); }
template <typename R> __host__ __device__ __forceinline__ Cx<R> operator-(Cx<R> a, Cx<R> b) { return Cx<R>(a.re - b.re, a.im - b.im); }
template <typename R> __host__ __device__ __forceinline__ Cx<R> operator-(Cx<R> a) { return Cx<R>(-a.re, -a.im); }
template <typename R> __host__ __device__ __forceinline__ Cx<R> operator*(Cx<R> a, Cx<R> b) {
  return Cx<R>(a.re * b.re - a.im * b.im, a.re * b.im + a.im * b.re);
}
template <typename R> __host__ __device__ __forceinline__ Cx<R> operator*(R s, Cx<R> a) { return Cx<R>(s * a.re, s * a.im); }
template <typename R> __host__ __device__ __forceinline__ Cx<R>& operator+=(Cx<R>& a, Cx<R> b) { a.re += b.re; a.im += b.im; return a; }
template <typename R> __host__ __device__ __forceinline__ Cx<R>& operator-=(Cx<R>& a, Cx<R> b) { a.re -= b.re; a.im -= b.im; return a; }
template <typename R> __host__ __device__ __forceinline__ Cx<R> conj(Cx<R> a) { return Cx<R>(a.re, -a.im); }
template <typename R> __host__ __device__ __forceinline__ R abs2(Cx<R> a) { return a.re * a.re + a.im * a.im; }
// acc += a * b (complex fused multiply-add)
template <typename R> __host__ __device__ __forceinline__ void cfma(Cx<R>& acc, Cx<R> a, Cx<R> b) {
  acc.re = fma(a.re, b.re, fma(-a.im, b.im, acc.re));
  acc.im = fma(a.re, b.im, fma(a.im, b.re, acc.im));
}
// acc += conj(a) * b
template <typename R> __host__ __device__ __forceinline__ void cfma_conj(Cx<R>& acc, Cx<R> a, Cx<R> b) {
  acc.re = fma(a.re, b.re, fma(a.im, b.im, acc.re));
  acc.im = fma(a.re, b.im, fma(-a.im, b.re, acc.im));
}
// ---- double <-> float by integer arithmetic ------------------------------------------------
// The FP64 unit of this GPU (half a lane a clock and scheduler) also serves the conversions:
// in the sweeps, those of r and z took longer than the multiply-adds.  Values in FP32's normal
// range (and zeros) are converted with integer operations, to the same bits.
__device__ __forceinline__ float to_float(double v) {
  const unsigned hi = (unsigned)__double2hiint(v), lo = (unsigned)__double2loint(v);
  const unsigned e = (hi >> 20) & 0x7ffu, sign = hi & 0x80000000u;
  if (e - 897u <= 253u) {               // 2^-126 <= |v| < 2^128: round to nearest even
    unsigned b = __funnelshift_l(lo, hi, 3) - 0xc0000000u;     // exponent bias 1023 -> 127
    b += ((lo & 0x1fffffffu) + 0x0fffffffu + (b & 1u)) >> 29;
    return __uint_as_float(b | sign);
  }
  if (e < 873u) return __uint_as_float(sign);                  // below half of the least subnormal
  return (float)v;
}
__device__ __forceinline__ double to_double(float v) {
  const unsigned b = __float_as_uint(v);
  if (((b >> 23) & 0xffu) - 1u <= 253u)
    return __hiloint2double((int)((b & 0x80000000u) | (((b & 0x7fffffffu) >> 3) + 0x38000000u)), (int)(b << 29));
  if ((b << 1) == 0u) return __hiloint2double((int)b, 0);
  return (double)v;
}
template <typename To, typename From> __host__ __device__ __forceinline__ Cx<To> cvt(Cx<From> a) {
#ifdef __CUDA_ARCH__
  if constexpr (sizeof(To) == 4 && sizeof(From) == 8) return Cx<To>(to_float(a.re), to_float(a.im));
  if constexpr (sizeof(To) == 8 && sizeof(From) == 4) return Cx<To>(to_double(a.re), to_double(a.im));
#endif
  return Cx<To>(To(a.re), To(a.im));
}
// 1 / a
template <typename R> __host__ __device__ __forceinline__ Cx<R> cinv(Cx<R> a) {
  R s = R(1) / (a.re * a.re + a.im * a.im);
  return Cx<R>(a.re * s, -a.im * s);
}

// principal square root
template <typename R> __host__ __device__ __forceinline__ Cx<R> csqrt(Cx<R> a) {
  R r = sqrt(a.re * a.re + a.im * a.im);
  R x = sqrt((r + a.re) * R(0.5));
  R y = sqrt((r - a.re) * R(0.5));
  return Cx<R>(x, a.im < 0 ? -y : y);
}

template <typename R> __device__ __forceinline__ Cx<R> shfl_xor(Cx<R> v, int off) {
  return Cx<R>(__shfl_xor_sync(0xffffffffu, v.re, off), __shfl_xor_sync(0xffffffffu, v.im, off));
}

// Sum of v[0..G) over the NL lanes that differ in the lane bits UNIT, 2 UNIT, ... NL/2 UNIT,
// scattered: each step a lane keeps half of its right-hand sides and hands the other half to
// its partner, so a lane ends with CNT = max(1, G / NL) sums, right-hand sides g .. g+CNT-1.
// With fewer right-hand sides than lanes the last steps are plain sums (every lane of such a
// group holds the same value; `first` marks one of them).
template <typename R, int G, int NL, int UNIT>
__device__ __forceinline__ void scatter_sum(Cx<R> (&v)[G], int lane, int& g, bool& first) {
  g = 0;
  first = true;
  int cnt = G;
#pragma unroll
  for (int o = NL / 2; o > 0; o >>= 1) {
    const bool up = (lane & (o * UNIT)) != 0;
    if (cnt > 1) {
      cnt >>= 1;
#pragma unroll
      for (int j = 0; j < G / 2; ++j)
        if (j < cnt) {
          const Cx<R> send = up ? v[j] : v[j + cnt];
          const Cx<R> keep = up ? v[j + cnt] : v[j];
          v[j] = keep + shfl_xor(send, o * UNIT);
        }
      if (up) g += cnt;
    } else {
      v[0] += shfl_xor(v[0], o * UNIT);
      first = first && !up;
    }
  }
}

// Reciprocal and reciprocal square root, in complex128 by two Newton steps from the FP32
// value (a handful of FP64 operations where the division and square root routines take
// dozens: a warp's FP64 instruction occupies its scheduler for about 64 clocks here)
__device__ __forceinline__ float rcp_of(float x) { return 1.0f / x; }
__device__ __forceinline__ double rcp_of(double x) {
  // for x well inside FP32's range
  double y = (double)(1.0f / (float)x);
  y = y * fma(-x, y, 2.0);
  return y * fma(-x, y, 2.0);
}
__device__ __forceinline__ float rsqrt_of(float x) { return rsqrtf(x); }
__device__ __forceinline__ double rsqrt_of(double x) {
  double y = (double)rsqrtf((float)x);
  const double h = 0.5 * x;
  y = y * fma(-h * y, y, 1.5);
  return y * fma(-h * y, y, 1.5);
}

// The same for any positive normal x: its exponent is taken out first.  All of them within 2^-51
// relative of the exact value (complex128).
__device__ __forceinline__ float rcp_any(float x) { return 1.0f / x; }
__device__ __forceinline__ float rsqrt_any(float x) { return 1.0f / sqrtf(x); }
__device__ __forceinline__ double rcp_any(double x) {
  const int e = min(((__double2hiint(x) >> 20) & 0x7ff) - 1023, 1022);
  const double s = __hiloint2double((1023 - e) << 20, 0);       // 2^-e (2^-1022 is the least normal)
  return rcp_of(x * s) * s;
}
__device__ __forceinline__ double rsqrt_any(double x) {
  const int q = (((__double2hiint(x) >> 20) & 0x7ff) - 1023) >> 1;
  const double s = __hiloint2double((1023 - q) << 20, 0);       // 2^-q
  return rsqrt_of(x * s * s) * s;
}
// The rotation of one-sided Jacobi for columns p, q with squared norms al, be (at least about
// 1e-28 of the largest column's) and inner product ga = <p, q>:
//     p' = cs p - conj(sne) q,  q' = cs q + sne p,  |p'|^2 = al - dn, |q'|^2 = be + dn.
// gg = |ga|^2 / (al be).  The angle comes from FP32 reciprocal square roots in both precisions
// (its error only leaves an inner product smaller by 1e-7, and the convergence does the rest);
// cs and the phase are refined to the storage precision.
template <typename R>
struct JacobiRotation {
  float gg, t;      // the squared cosine; the tangent
  R cs, dn;
  Cx<R> sne;
  __device__ __forceinline__ bool needed(R al, R be, Cx<R> ga, float tol2) {
    s = R(rsqrtf((float)al)) * R(rsqrtf((float)be));
    gn = s * ga;
    gg = (float)abs2(gn);
    return gg > tol2;
  }
  __device__ __forceinline__ void angle(R al, R be) {
    const float ig = rsqrtf(gg);
    const float z = 0.5f * (float)((be - al) * s) * ig;
    // (z reaches 1e29 in complex128, where its square would overflow)
    const float za = fabsf(z);
    t = copysignf(1.0f, z) / (za + (za < 1e9f ? sqrtf(fmaf(z, z, 1.0f)) : za));
    const R tr = (R)t;
    cs = rsqrt_of(fma(tr, tr, R(1)));
    R igr = (R)ig;
    if (sizeof(R) == 8) igr = igr * fma(R(-0.5) * abs2(gn) * igr, igr, R(1.5));
    sne = (tr * cs * igr) * gn;
    dn = tr * (abs2(gn) * igr * rcp_of(s));
  }

 private:
  R s;
  Cx<R> gn;
};

// One-sided Jacobi ends after a sweep whose cosines were all small (1e-4 in complex64, 1e-8 in
// complex128), if its rotations cannot have left more than the orthogonality tolerance: a rotation
// by tan t mixes the other inner products of its two columns, so up to t times the largest cosine
// is left, t being small between well-separated singular values (the quadratic convergence) but
// not within a cluster.  gg: the largest squared cosine, t: the largest tangent, tol2: the squared tolerance.
__device__ __forceinline__ bool rotations_done(float gg, float t, float tol2) {
  return t * sqrtf(gg) <= 2.0f * sqrtf(tol2);
}

// L2-only loads/stores for data exchanged between CTAs of one sweep team.
template <typename R> __device__ __forceinline__ Cx<R> ld_cg(const Cx<R>* p);
template <> __device__ __forceinline__ Cx<float> ld_cg(const Cx<float>* p) {
  float2 v = __ldcg(reinterpret_cast<const float2*>(p)); return Cx<float>(v.x, v.y);
}
template <> __device__ __forceinline__ Cx<double> ld_cg(const Cx<double>* p) {
  double2 v = __ldcg(reinterpret_cast<const double2*>(p)); return Cx<double>(v.x, v.y);
}
template <typename R> __device__ __forceinline__ void st_cg(Cx<R>* p, Cx<R> v);
template <> __device__ __forceinline__ void st_cg(Cx<float>* p, Cx<float> v) {
  __stcg(reinterpret_cast<float2*>(p), make_float2(v.re, v.im));
}
template <> __device__ __forceinline__ void st_cg(Cx<double>* p, Cx<double> v) {
  __stcg(reinterpret_cast<double2*>(p), make_double2(v.re, v.im));
}

// Device status word: [0] = first error code (HSWEEP_ERR_*), [1] = layer.
__device__ __forceinline__ void report_error(int* status, int code, int layer) {
  if (status && atomicCAS(status, 0, code) == 0) status[1] = layer;
}

#define HSW_CUDA(call)                                   \
  do {                                                   \
    cudaError_t e_ = (call);                             \
    if (e_ != cudaSuccess) return HSWEEP_ERR_CUDA;       \
  } while (0)

static inline unsigned div_up(long long a, long long b) { return unsigned((a + b - 1) / b); }
