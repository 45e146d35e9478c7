// FP64-accurate complex GEMM from integer BF16 slices on the tensor cores; see tc_slice.cu.
#pragma once

#include <vector>

#include "tc_gemm.cuh"

namespace adc {

// significant bits of an FP64 product (eight digits): operand rounding 2^-57 and dropped
// classes of about 2^-58 of the row and column maxima
constexpr int kDigitFp64Bits = 56;

constexpr int SL_DIGIT = 7;  // bits of a digit, but for the setup's products (sl_digits)
// digits of an operand: ns of b bits
struct SlDigits {
  int b, ns;
};
// Seven-bit digits, the widest whose products FP32 sums exactly over useful runs (eight-bit
// ones drain four times as often): 4, 6 and 8 of them for about 24, 40 and 56 bits.
// The setup's 48-bit products take digits whose whole inner sum fits FP32 (b = 7 .. 4
// as the inner size grows): which bits of the operators they keep depends on the
// digits, and the BF16 split of an operator must not change with how it was computed.
inline SlDigits sl_digits(int64_t K, int bits) {
  int b = SL_DIGIT;
  if (bits > 40 && bits < kDigitFp64Bits) {
    const int64_t K2 = K <= 0 ? 128 : (K + 63) / 64 * 128;
    int l = 0;
    while ((1ll << l) < K2) ++l;
    b = (24 - l) / 2;
    b = b < 4 ? 4 : b > 7 ? 7 : b;
  }
  return {b, (bits + b - 1) / b};
}
// inner size as stored: padded to whole blocks of 64
inline int64_t sl_kp(int64_t K) { return K <= 0 ? 64 : (K + 63) / 64 * 64; }

// An operand as ns BF16 planes of integer digits, [rows][2*kp] each, and one
// scale per row (A: per row; B: per complex row, shared by its two embedded
// rows): the largest magnitude's leading word, see tc_slice.cu.
struct SlMat {
  DBuf planes, exps;
  int b = 0, ns = 0;
  int64_t rows = 0, kp = 0, kreal = 0;
};

// scratch of sl_gemm: the per-CTA spill of the less significant classes and
// the partial products of a split inner index
struct SlWork {
  DBuf spill, part;
};

// digits of a context's static operators (A side), each built when a product first needs
// it, and the per-call B operand: shared by the sliced products (their leading digits) and
// the FP64 ones
enum { SL_CPL = 0, SL_CPLT = 1, SL_GLAD = 2, SL_W = 3, SL_NOPS = 4 };
struct SlCache {
  SlMat op[SL_NOPS], Bx;
  int rest[SL_NOPS] = {};  // FP64 products of the operator left before its digits may be built again
  SlWork w;
  DBuf err;
  Exec &ex;
  const int dev;
  int busy = 0;       // a product is being enqueued: its operator's digits stay
  double kept = 0.0;  // bytes of digits kept for FP64 products alone
  SlCache(Exec &e, int d);
  ~SlCache();
};

// A[m][k] = op(src[m*s_m + k*s_k]); digits for about `bits` significant bits, with cut_from
// the leading digits of the slicing to that many bits
void sl_pack_A(Exec &ex, SlMat &dst, const cplx *src, int64_t M, int64_t K, int64_t s_m, int64_t s_k, bool conj,
               int bits, int cut_from = 0);
// B[n][k] = op(src[(n / n_in)*s_nh + (n % n_in)*s_nl + k*s_k]), sliced like the A operand `like`
// bits > 0: only the leading digits for about that many significant bits (the
// product then uses the same leading slices of A)
void sl_pack_B(Exec &ex, SlMat &dst, const cplx *src, int64_t Nc, int64_t K, int64_t s_nh, int64_t s_nl,
               int64_t n_in, int64_t s_k, bool conj, const SlMat &like, int bits = 0);
// B operand of the ring term, gathered from the packed satellite block of X
void sl_pack_B_ring(Exec &ex, SlMat &dst, const adc_ctx *c, const cplx *X, int64_t k, const SlMat &like,
                    int bits = 0);
// zgemm's contract (tensor.cuh) computed as the sliced product with ex.sliced_bits bits
void zgemm_sliced(Exec &ex, int64_t M, int64_t N, int64_t K, int64_t batch, cplx alpha, const cplx *A, int64_t sAb,
                  int64_t sAm, int64_t sAk, bool conjA, const cplx *B, int64_t sBb, int64_t sBk, int64_t sBn,
                  bool conjB, cplx beta, cplx *C, int64_t sCb, int64_t sCm, int64_t sCn);
// zgemm's FP64 product of a large shape from 56-bit digits, asynchronous; false when it
// is left to the FP64 units (small, under stream capture, no room for the digit planes).
// A wait that gave up leaves NaN in the output and its code in *ex.digit_err
bool zgemm_fp64_digits(Exec &ex, int64_t M, int64_t N, int64_t K, int64_t batch, cplx alpha, const cplx *A,
                       int64_t sAb, int64_t sAm, int64_t sAk, bool conjA, const cplx *B, int64_t sBb, int64_t sBk,
                       int64_t sBn, bool conjB, cplx beta, cplx *C, int64_t sCb, int64_t sCm, int64_t sCn);
// whether an FP64 product of this shape would run from digits now (size, not under capture)
bool fp64_digits_usable(Exec &ex, int64_t M, int64_t N, int64_t K);
// out = alpha A B^T + beta out, addressing as tc_gemm
void sl_gemm(Exec &ex, const SlMat &A, const SlMat &B, int64_t M, int64_t N, cplx alpha, cplx beta, cplx *out,
             int64_t s_m, int64_t s_nh, int64_t s_nl, int64_t n_in, int *err, SlWork &w);

// pipeline wait limit of this file's kernels (tc_set_wait_ns sets both files')
void sl_set_wait_ns(unsigned long long ns);
// test hook: bytes per operand chunk of zgemm_sliced (0 restores the free-memory rule)
void set_sliced_cap_bytes(size_t bytes);

}  // namespace adc
