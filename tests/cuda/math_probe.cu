// The functions of hr_math.cuh on arrays of bit patterns, beside the language's
// operations (tests/test_gpu_math.py builds and loads this file).
#include "hr_math.cuh"

namespace {

enum { RCP, SQRT, RSQRT, SQRT_OF_PAIR, RSQRT_OF_PAIR, NARROW, WIDEN };

__global__ void k_probe(int op, int own, int n, const unsigned long long* __restrict__ in,
                        unsigned long long* __restrict__ out) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const double x = __longlong_as_double((long long)in[i]);
    double r = 0.0, y = 0.0;
    if (op == RCP) y = own ? hr::rcp(x) : 1.0 / x;
    if (op == SQRT) y = own ? hr::sqrt64(x) : sqrt(x);
    if (op == RSQRT) y = own ? hr::rsqrt64(x) : 1.0 / sqrt(x);
    if (op == SQRT_OF_PAIR) y = own ? hr::sqrt_rsqrt(x, &r) : sqrt(x);
    if (op == RSQRT_OF_PAIR) {
      if (own) hr::sqrt_rsqrt(x, &r);
      y = own ? r : 1.0 / sqrt(x);
    }
    if (op == NARROW) {
      out[i] = __float_as_uint(own ? hr::narrow(x) : (float)x);
      continue;
    }
    if (op == WIDEN) {
      const float f = __uint_as_float((unsigned)in[i]);
      y = own ? hr::widen(f) : (double)f;
    }
    out[i] = (unsigned long long)__double_as_longlong(y);
  }
}

}  // namespace

extern "C" int math_probe(int op, int own, int n, const void* in, void* out, void* stream) {
  k_probe<<<256, 256, 0, (cudaStream_t)stream>>>(op, own, n, (const unsigned long long*)in, (unsigned long long*)out);
  return (int)cudaGetLastError();
}
