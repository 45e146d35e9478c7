// Shared definitions of the GB300 ADC library (host and device).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <cstdio>
#include <stdexcept>
#include <string>
#include <vector>

#include "../../include/adc_gb300.h"

namespace adc {

typedef double2 cplx;  // interleaved (re, im), the layout of adc_c128

// Error carried from deep inside the setup code to the ABI boundary, where it
// becomes a negative return code. Nothing below the boundary aborts.
struct Error : public std::runtime_error {
  int code;
  Error(int c, const std::string &m) : std::runtime_error(m), code(c) {}
};

#define ADC_CUDA(call)                                                           \
  do {                                                                           \
    cudaError_t e_ = (call);                                                     \
    if (e_ != cudaSuccess)                                                       \
      throw ::adc::Error(ADC_ERR_CUDA, std::string(#call) + ": " +              \
                                           cudaGetErrorString(e_) + " at " +     \
                                           __FILE__ + ":" + std::to_string(__LINE__)); \
  } while (0)

// every kernel launch site calls ADC_CHECK_LAUNCH(), which also counts it
extern long long g_launches;
#define ADC_CHECK_LAUNCH()                               \
  do {                                                   \
    __atomic_add_fetch(&::adc::g_launches, 1, __ATOMIC_RELAXED); \
    ADC_CUDA(cudaGetLastError());                        \
  } while (0)

#define ADC_REQUIRE(cond, code, msg)                 \
  do {                                               \
    if (!(cond)) throw ::adc::Error((code), (msg));  \
  } while (0)

__host__ __device__ inline cplx cmake(double r, double i) { return make_double2(r, i); }
__host__ __device__ inline cplx cadd(cplx a, cplx b) { return make_double2(a.x + b.x, a.y + b.y); }
__host__ __device__ inline cplx csub(cplx a, cplx b) { return make_double2(a.x - b.x, a.y - b.y); }
__host__ __device__ inline cplx cmul(cplx a, cplx b) {
  return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
__host__ __device__ inline cplx cconj(cplx a) { return make_double2(a.x, -a.y); }
__host__ __device__ inline cplx cscale(cplx a, double s) { return make_double2(a.x * s, a.y * s); }
// acc += a * b
__host__ __device__ inline void cfma(cplx &acc, cplx a, cplx b) {
  acc.x = fma(a.x, b.x, acc.x);
  acc.x = fma(-a.y, b.y, acc.x);
  acc.y = fma(a.x, b.y, acc.y);
  acc.y = fma(a.y, b.x, acc.y);
}

// A factor by kind: 0 zero, 1 one, 2 real, 3 complex. The element-wise kernels take the
// kind, because a complex multiply by 1 or by a real factor costs four FP64 operations of
// which none or two are needed, and at two a clock and SM they, not memory, bound such kernels.
inline int factor_kind(cplx a) { return a.y != 0.0 ? 3 : a.x == 1.0 ? 1 : a.x == 0.0 ? 0 : 2; }
__device__ __forceinline__ cplx scaled(int kind, cplx a, cplx v) {
  if (kind == 1) return v;
  if (kind == 3) return cmul(a, v);
  return make_double2(a.x * v.x, a.x * v.y);
}
// alpha v + beta *old
__device__ __forceinline__ cplx axpby(int ka, cplx alpha, cplx v, int kb, cplx beta, const cplx *old) {
  cplx r = scaled(ka, alpha, v);
  if (kb) {
    const cplx o = scaled(kb, beta, *old);
    r = make_double2(r.x + o.x, r.y + o.y);
  }
  return r;
}

// Division of n < 2^31 by a constant found at run time (Granlund and Montgomery, "Division by
// invariant integers using multiplication", 1994): two multiplies' worth instead of
// the tens of instructions of an integer division
struct FastDiv {
  uint32_t d, mul, sh;
};
inline FastDiv fast_div(uint32_t d) {
  FastDiv f{d, 1, 0};
  while ((1ull << f.sh) < d) ++f.sh;
  f.mul = (uint32_t)((((1ull << f.sh) - d) << 32) / d + 1);
  return f;
}
__device__ __forceinline__ uint32_t fdiv(uint32_t n, FastDiv f) { return (__umulhi(n, f.mul) + n) >> f.sh; }

// index of the pair (p < q) among the n(n-1)/2 pairs, row-major upper triangle
__host__ __device__ inline int64_t pair_index(int64_t p, int64_t q, int64_t n) {
  return p * n - p * (p + 1) / 2 + (q - p - 1);
}

inline int64_t npairs(int64_t n) { return n * (n - 1) / 2; }

inline unsigned grid1d(int64_t n, int threads) {
  int64_t b = (n + threads - 1) / threads;
  if (b > (int64_t)1 << 30) b = (int64_t)1 << 30;
  if (b < 1) b = 1;
  return (unsigned)b;
}

}  // namespace adc
