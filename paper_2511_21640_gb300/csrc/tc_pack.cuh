// Tiles of a complex operand read for packing (BF16 planes of tc_gemm.cu, digits of
// tc_slice.cu): 32 rows by 64 inner elements per block of 256 threads, read with
// lanes along whichever index is contiguous in memory.
#pragma once

#include "tc_gemm.cuh"

namespace adc {

namespace {

constexpr int PK_R = 32, PK_K = 64;    // tile of the packing kernels: rows x inner elements
constexpr int PK_LD = PK_K + PK_K / 8;  // one element of padding per eight
__device__ __forceinline__ int pk_at(int r, int k) { return r * PK_LD + k + (k >> 3); }

// element (row n, inner k) of the operand rows a packing block handles: the
// address arithmetic of BSrc split into a part per row and a part per k
struct PkRow {
  const cplx *p;
  int b;
};
__device__ __forceinline__ PkRow pk_row(const BSrc &s, int64_t n) {
  PkRow r;
  if (s.mode == 0) {
    const int64_t nh = n / s.n_in, nl = n - nh * s.n_in;
    r.p = s.p + nh * s.s_nh + nl * s.s_nl;
    r.b = 0;
  } else {
    const int64_t per = (s.mode == 1) ? s.v : s.o, vec = n / per;
    r.p = s.p + s.n1 + vec * s.N;
    r.b = (int)(n - vec * per);
  }
  return r;
}
__device__ __forceinline__ cplx pk_get(const BSrc &s, const PkRow &r, int64_t k, int kh, int kl) {
  if (s.mode == 0) return r.p[k * s.s_k];
  // the pair (p < q) of n at p n - p (p + 1) / 2 + q - p - 1 (32 bits reach 46340 spinors)
  const bool ea = (s.mode == 1);  // (kh, kl) = (kk, c): X[kk][(c, b)]; else (kq, b): X[(i, kq)][b]
  const int j = ea ? kl : kh, n = (int)(ea ? s.v : s.o);
  if (j == r.b) return cmake(0.0, 0.0);
  const int p = min(j, r.b), q = max(j, r.b);
  const int pair = p * n - p * (p + 1) / 2 + q - p - 1;
  const cplx x = ea ? r.p[(int64_t)kh * (n * (n - 1) / 2) + pair] : r.p[(int64_t)pair * s.v + kl];
  return (ea ? j < r.b : r.b < j) ? x : cmake(-x.x, -x.y);
}

// loads rows [n0, n0 + 32) x [k0, k0 + 64) of the source, zero outside, calling
// f(row, k, value); lanes run along whichever index is contiguous in memory
template <class F>
__device__ __forceinline__ void pk_load(const BSrc &src, int64_t n0, int64_t rows, int64_t k0, int64_t K, bool kfast,
                                        const PkRow *row, F f) {
  // a thread keeps its inner element (or its row) over the steps
  if (kfast) {
    const int kk = threadIdx.x & 63;
    const int64_t k = k0 + kk;
    int kh = 0, kl = 0;
    if (src.mode != 0) { kh = (int)((unsigned)k / (unsigned)src.v); kl = (int)k - kh * (int)src.v; }
#pragma unroll
    for (int it = 0; it < PK_R * PK_K / 256; ++it) {
      const int r = (threadIdx.x >> 6) + 4 * it;
      f(r, kk, n0 + r < rows && k < K ? pk_get(src, row[r], k, kh, kl) : cmake(0.0, 0.0));
    }
  } else {  // strided sources only (pk_kfast)
    const int r = threadIdx.x & 31;
#pragma unroll
    for (int it = 0; it < PK_R * PK_K / 256; ++it) {
      const int kk = (threadIdx.x >> 5) + 8 * it;
      const int64_t k = k0 + kk;
      f(r, kk, n0 + r < rows && k < K ? pk_get(src, row[r], k, 0, 0) : cmake(0.0, 0.0));
    }
  }
}

}  // namespace

// lanes along the inner index, unless only the row index is contiguous
inline int pk_kfast(const BSrc &s) { return (s.mode != 0 || s.s_k == 1 || s.s_nl != 1) ? 1 : 0; }

}  // namespace adc
