// C entry points that apply the scalar helpers of csrc/common.cuh to arrays, for tests/test_gpu_scalars.py.
#include "../../paper_1007_4290_gb300/csrc/common.cuh"
#include "dev.cuh"

namespace {

template <typename T, typename F>
__global__ void map(int n, const T* in, F* out, int op) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const T x = in[i];
  if constexpr (sizeof(T) == 8 && sizeof(F) == 4) {
    out[i] = op ? (float)x : to_float(x);
  } else if constexpr (sizeof(T) == 4) {
    out[i] = op ? (double)x : to_double(x);
  } else {
    out[i] = op == 0 ? rcp_of(x) : op == 1 ? rsqrt_of(x) : op == 2 ? rcp_any(x) : rsqrt_any(x);
  }
}

template <typename T, typename F>
int apply(int n, const T* in, F* out, int op) {
  Dev<T> a(n, in);
  Dev<F> b(n);
  if (!a.p || !b.p) return 2;
  map<T, F><<<(n + 255) / 256, 256>>>(n, a.p, b.p, op);
  return cudaDeviceSynchronize() == cudaSuccess && b.get(out) ? 0 : 4;
}

}  // namespace

// op 0: the library's conversion, 1: the compiler's
ENTRY narrow(int n, const double* in, float* out, int op) { return apply(n, in, out, op); }
ENTRY widen(int n, const float* in, double* out, int op) { return apply(n, in, out, op); }
// op 0: rcp_of, 1: rsqrt_of, 2: rcp_any, 3: rsqrt_any
ENTRY newton(int n, const double* in, double* out, int op) { return apply(n, in, out, op); }
