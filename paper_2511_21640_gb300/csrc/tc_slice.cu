// FP64-accurate complex GEMM from BF16 slices on the tensor cores.
//
// out[m][n] = alpha * sum_k A[m][k] B[n][k] + beta * out[m][n]   (complex)
//
// The operands use the real embedding of tc_gemm.cu (an A row is [Re | Im], a
// complex B row n becomes [Re | -Im] and [Im | Re]). Every row of an operand
// is scaled by a power of two, 2^E with max |row| < 2^E, and each scaled value
// y (|y| < 1), rounded to a multiple of 2^(-b ns), is written with ns signed
// digits of b bits (seven, but see sl_digits), y = sum_i d_i 2^(-b i), |d_1| <= 2^b
// and |d_i| <= 2^(b-1) after it: integers that BF16 holds exactly. A product of digit i of A and
// digit j of B has weight 2^(-b (i + j)); the pairs of one weight form a class
// c = i + j, and the classes 2 .. ns + 1 are kept. The error comes only from
// the rounding of the operands and the dropped classes, about 2^(-b ns)
// relative to the row and column maxima, whatever K is: an error-free
// splitting of the products in the manner of Ozaki, Ogita, Oishi and Rump
// ("Error-free transformations of matrix multiplication by using fast
// routines of matrix multiplication", Numer. Algorithms 59, 2012), on BF16
// tensor cores with integer digits.
//
// Exactness. All pairs of one class add into the same FP32 accumulator. Per
// inner element a class of n pairs adds at most (n + 2) 2^(2b-2) in magnitude (two
// of its pairs hold a first digit; the class of the pair (1, 1) alone at most
// 2^(2b) = 4 * 2^(2b-2)), so a run of floor(2^(20-2b) / (n + 2)) blocks of 64 stays
// within 2^24 and every partial sum is an integer that FP32 holds. After such a
// run the accumulators are drained into 64-bit integers.
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>

#include "ctx.cuh"
#include "tc_gemm.cuh"
#include "tc_pack.cuh"
#include "tc_ptx.cuh"
#include "tc_slice.cuh"

namespace adc {

namespace {

// ---------------------------------------------------------------- row scales
// The scale of a row is kept as one word: the high 31 bits of its largest |x| with 64 added to
// the exponent field; b + 12 in that field when it is subnormal and has b significant bits.
// 0: a row of zeros; the field kWordInf: the row holds an infinity or a NaN. The exponent
// E follows by one subtraction (the product's results take it per column).
constexpr unsigned kWordInf = 0x7ffu + 64u;
// high 31 bits of |x|, the lowest bit set too when only the low word is nonzero: an integer
// maximum finds the largest but among subnormal numbers (below 0x100000)
__device__ __forceinline__ unsigned mag_word(double x) {
  const unsigned hi = (unsigned)__double2hiint(x) & 0x7fffffffu;
  return hi | (__double2loint(x) != 0 ? 1u : 0u);
}
__device__ __forceinline__ unsigned mag_word(cplx x) { return max(mag_word(x.x), mag_word(x.y)); }
// the row's word for a subnormal x (zero: 0)
__device__ __forceinline__ unsigned subnormal_word(double x) {
  const long long m = __double_as_longlong(x) & 0x7fffffffffffffffll;
  return m ? (unsigned)(64 - __clzll(m) + 12) << 20 : 0u;
}
__device__ __forceinline__ bool not_finite(unsigned w) { return (w >> 20) == kWordInf; }
// E with every |x| of the row below 2^E, and 2^E at most twice the largest (any E for zeros)
__device__ __forceinline__ int scale_exp(unsigned w) { return (int)(w >> 20) - 1086; }

// round(x 2^(bits - E)) as an integer (|x| < 2^E, so at most 2^bits; ties to even)
__device__ __forceinline__ long long fixed_of(double x, int E, int bits) {
  const long long u = __double_as_longlong(x);
  const int field = (int)((u >> 52) & 0x7ff);
  long long m = u & 0xfffffffffffffll;
  if (field) m |= 1ll << 52;
  const int s = (field ? field : 1) - 1075 + bits - E;  // value = m 2^(s + E - bits), m 2^s < 2^bits
  long long r;
  if (s >= 0) r = m << s;
  else if (s >= -54) r = (m + ((1ll << (-s - 1)) - 1) + ((m >> -s) & 1)) >> -s;
  else r = 0;
  return u < 0 ? -r : r;
}

// W[n] = max(W[n], largest magnitude word of row n over the inner range of this
// block). Blocks: (row tiles, inner ranges); the maximum is exact in any order
__global__ void __launch_bounds__(256)
k_sl_scale(BSrc src, int64_t rows, int64_t K, int64_t krange, int kfast, unsigned *W) {
  __shared__ PkRow row[PK_R];
  __shared__ unsigned mx[PK_R];
  const int64_t kb = (int64_t)blockIdx.y * krange, ke = min(K, kb + krange);
  for (int64_t n0 = (int64_t)blockIdx.x * PK_R; n0 < rows; n0 += (int64_t)gridDim.x * PK_R) {
    if (threadIdx.x < PK_R) {
      row[threadIdx.x] = pk_row(src, min(n0 + (int64_t)threadIdx.x, rows - 1));
      mx[threadIdx.x] = 0;
    }
    __syncthreads();
    unsigned own = 0;  // lanes along the rows: one row per thread
    for (int64_t k0 = kb; k0 < ke; k0 += PK_K)
      pk_load(src, n0, rows, k0, ke, kfast != 0, row, [&](int r, int, cplx x) {
        const unsigned w = mag_word(x);
        if (kfast) {
          const unsigned m = __reduce_max_sync(0xffffffffu, w);  // a warp covers half a row
          if ((threadIdx.x & 31) == 0) atomicMax(&mx[r], m);
        } else {
          own = max(own, w);
        }
      });
    if (!kfast) atomicMax(&mx[threadIdx.x & 31], own);
    __syncthreads();
    const unsigned top = threadIdx.x < PK_R ? mx[threadIdx.x] : 0;
    unsigned word = top >= 0x100000u ? top + (64u << 20) : 0;
    // rows of subnormal numbers here: once more, by their significant bits (a branch among the
    // loads above would keep them from overlapping)
    if (__syncthreads_or(top != 0 && top < 0x100000u)) {
      if (threadIdx.x < PK_R) mx[threadIdx.x] = 0;
      __syncthreads();
      for (int64_t k0 = kb; k0 < ke; k0 += PK_K)
        pk_load(src, n0, rows, k0, ke, kfast != 0, row, [&](int r, int, cplx x) {
          if (mag_word(x) < 0x100000u) atomicMax(&mx[r], max(subnormal_word(x.x), subnormal_word(x.y)));
        });
      __syncthreads();
      if (threadIdx.x < PK_R && top < 0x100000u) word = mx[threadIdx.x];
    }
    if (threadIdx.x < PK_R && n0 + threadIdx.x < rows) atomicMax(&W[n0 + threadIdx.x], word);
    __syncthreads();
  }
}

__device__ __forceinline__ uint32_t bf16x2_of(int a, int b) {
  const __nv_bfloat162 h = __floats2bfloat162_rn((float)a, (float)b);  // exact: |a|, |b| <= 128
  return *(const uint32_t *)&h;
}

// Bound by memory (16 bytes read, 4 ns or 8 ns written per element); the tile in
// shared memory lets lanes run along whichever source index is contiguous.
// Digits of a 32 x 64 tile staged in shared memory: every thread takes eight
// consecutive inner elements of a row and stores 16 bytes per plane. EMB = 1:
// an A row [Re | Im]; EMB = 2: the two rows of the B embedding.
// The digits come from the top, each the remainder rounded to nearest, so that
// they are centred on zero: digits cut from the bottom, in [-2^(b-1), 2^(b-1) - 1],
// have a mean of -1/2, and the dropped classes would leave an error that grows with K.
// bits: of the integer they are cut from, b ns or more (then these are its leading digits).
template <int EMB>
__global__ void __launch_bounds__(256)
k_sl_pack(BSrc src, int64_t rows, int64_t K, int conj, int64_t kp, int kfast, const unsigned *__restrict__ W, int b, int ns,
          int bits, __nv_bfloat16 *base, int64_t pe) {
  __shared__ cplx tile[PK_R * PK_LD];
  __shared__ PkRow row[PK_R];
  for (int64_t n0 = (int64_t)blockIdx.x * PK_R; n0 < rows; n0 += (int64_t)gridDim.x * PK_R) {
    if (threadIdx.x < PK_R) row[threadIdx.x] = pk_row(src, min(n0 + (int64_t)threadIdx.x, rows - 1));
    __syncthreads();
    for (int64_t k0 = (int64_t)blockIdx.y * PK_K; k0 < kp; k0 += (int64_t)gridDim.y * PK_K) {
      pk_load(src, n0, rows, k0, K, kfast != 0, row, [&](int r, int kk, cplx x) { tile[pk_at(r, kk)] = x; });
      __syncthreads();
      const int r = threadIdx.x >> 3, oct = threadIdx.x & 7;
      const int64_t n = n0 + r;
      if (n < rows) {
        const unsigned w = W[n];
        const int e = scale_exp(w);
        const bool dead = w == 0 || not_finite(w);
        long long re[8], im[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const cplx x = tile[pk_at(r, 8 * oct + j)];
          re[j] = dead ? 0 : fixed_of(x.x, e, bits);
          im[j] = dead ? 0 : fixed_of(conj ? -x.y : x.y, e, bits);
        }
        for (int i = 0; i < ns; ++i) {
          const int sh = bits - b * (i + 1);
          const long long rnd = (1ll << sh) >> 1;
          int dr[8], di[8];
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            dr[j] = (int)((re[j] + rnd) >> sh);
            di[j] = (int)((im[j] + rnd) >> sh);
            re[j] -= (long long)dr[j] << sh;
            im[j] -= (long long)di[j] << sh;
          }
          uint4 vr, vi;
          vr.x = bf16x2_of(dr[0], dr[1]); vr.y = bf16x2_of(dr[2], dr[3]);
          vr.z = bf16x2_of(dr[4], dr[5]); vr.w = bf16x2_of(dr[6], dr[7]);
          vi.x = bf16x2_of(di[0], di[1]); vi.y = bf16x2_of(di[2], di[3]);
          vi.z = bf16x2_of(di[4], di[5]); vi.w = bf16x2_of(di[6], di[7]);
          __nv_bfloat16 *pl = base + (int64_t)i * pe + (int64_t)EMB * n * 2 * kp + k0 + 8 * oct;
          *(uint4 *)pl = vr;
          if (EMB == 1) {
            *(uint4 *)(pl + kp) = vi;
          } else {
            uint4 vn;
            vn.x = bf16x2_of(-di[0], -di[1]); vn.y = bf16x2_of(-di[2], -di[3]);
            vn.z = bf16x2_of(-di[4], -di[5]); vn.w = bf16x2_of(-di[6], -di[7]);
            *(uint4 *)(pl + kp) = vn;
            *(uint4 *)(pl + 2 * kp) = vi;
            *(uint4 *)(pl + 3 * kp) = vr;
          }
        }
      }
      __syncthreads();
    }
  }
}

// ---------------------------------------------------------------- the product
// One CTA per SM, resident, takes output tiles of 128 rows by BN real columns.
// Four classes c = hi, hi - 1, .. share a pass over K with one TMEM accumulator
// each (4 x BN columns); stage i of an inner block holds digit i of A and digit
// hi - i of B, and digit hi - i of B is multiplied with the digits i, i - 1, ..
// of A, which are still in shared memory from the stages before. So a pass of
// the classes 9..6 reads 16 operand blocks for 26 block products, where one
// product at a time reads 52: a 128 x 128 x 64 block product takes 256 clocks
// of the tensor core and 32 KB from L2, 128 bytes a clock for every SM, far
// more than L2 delivers; shared, it is 39.
// Warp 0 issues the TMA loads, warp 1 the MMAs, warps 2..9 drain the
// accumulators (integer multiply-adds; the FP64 units would take longer than
// the MMAs) and form the results from 128-bit integers, rounded once, while
// the next tile's MMAs run. The passes run from the least significant classes
// up; the first one's sums wait in a global buffer per CTA (L2).
// What bounds it: the tensor cores, and at short inner sizes forming the results.
// Measured (GB300, 40-bit digits ready, M x N x K complex), with every digit pair a
// product of its own, FP32 sums through memory and a combining kernel, then now:
// 19900 x 320 x 19900 48.1 -> 13.3 ms (1.60 PFLOP/s of BF16 products), 8100 x 8100 x 540
// 4.9 ms (1.2 PFLOP/s: results and drains weigh more), 180 x 6 x 402752 0.62 ms.
struct SlArgs {
  CUtensorMap mA, mB;
  int M, N2, b, ns, kps, kb_per_split, ksplit, tiles_m, tiles_n, panel, items;
  const unsigned *WA, *WB;
  cplx *out;
  int64_t s_m, s_nh, s_nl;
  int n_in, amode, bmode;  // amode, bmode: 0 the factor is 1 (alpha) or 0 (beta), 1 real, 2 complex
  cplx alpha, beta;
  cplx *part;         // [ksplit][M][N2 / 2] partial products when ksplit > 1
  long long *spill;   // [CTA][BN / H][32 * 4 H]
  int *err;
};

template <int BN>
struct SlTile {
  static constexpr int ABYTES = 128 * 64 * 2, BBYTES = BN * 64 * 2, STAGE = ABYTES + BBYTES;
  static constexpr int ST = BN == 128 ? 7 : BN == 64 ? 9 : 11;
  static constexpr int BAR_OFF = ST * STAGE;
  static constexpr int SMEM = 1024 + BAR_OFF + 256;
  static constexpr int H = BN >= 64 ? 2 : 1;  // column halves, four draining warps each
  static constexpr int VALS = BN / H;         // values per draining thread
  static constexpr uint32_t TMEM_COLS = 4 * BN;
};

struct SlItem {
  int m0, n0, split, kb_beg, kb_end;
};
template <int BN>
__device__ __forceinline__ SlItem sl_item(const SlArgs &a, int it) {
  SlItem d;
  const int tiles = a.tiles_m * a.tiles_n;
  d.split = it / tiles;
  const int t = it - d.split * tiles;
  // panels of a.panel column tiles; row tiles inside a panel, columns fastest
  const int full = (a.tiles_n / a.panel) * a.panel * a.tiles_m;
  int w = a.panel, p = 0, r = t;
  if (t < full) {
    p = t / (a.panel * a.tiles_m);
    r = t - p * (a.panel * a.tiles_m);
  } else {
    p = a.tiles_n / a.panel;
    r = t - full;
    w = a.tiles_n - p * a.panel;
  }
  const int tm = r / w;
  d.m0 = tm * 128;
  d.n0 = (p * a.panel + r - tm * w) * BN;
  d.kb_beg = d.split * a.kb_per_split;
  d.kb_end = min(a.kps, d.kb_beg + a.kb_per_split);
  return d;
}

// highest class of a pass, classes of the pass, inner blocks per exact run
__device__ __forceinline__ int pass_classes(int hi) { return min(4, hi - 1); }
__device__ __forceinline__ int pass_run(int hi, int b) { return (1 << (20 - 2 * b)) / (hi == 2 ? 4 : hi + 1); }

// (hi 2^sh + lo) 2^e rounded to nearest: hi is shifted up as far as 64 bits allow (62 bits
// of the sum at least are kept), the sum normalised and packed with integer instructions
__device__ __forceinline__ double scaled_sum(long long hi, int sh, long long lo, int e) {
  const int room = max(0, __clzll(hi < 0 ? -hi : hi) - 2);
  const int up = min(sh, room);
  const long long v = (long long)((unsigned long long)hi << up) + (lo >> (sh - up));
  unsigned long long u = (unsigned long long)(v < 0 ? -v : v);
  if (u == 0) return 0.0;
  const int lz = __clzll((long long)u);
  u <<= lz;
  const unsigned long long m = (u >> 11) + ((u >> 10) & 1);  // 53 bits, the leading one set (or 2^53)
  const int be = 63 - lz + (sh - up) + e + 1023;
  if (be < 1 || be > 2045) {
    const double r = ldexp((double)m, be - 1075);
    return v < 0 ? -r : r;
  }
  return __longlong_as_double((long long)((((unsigned long long)(be - 1) << 52) + m) |
                                          ((unsigned long long)v & 0x8000000000000000ull)));
}

// The same in two FP64 operations where hi 2^sh + lo = H 2^sh + L with |H| < 2^51 and
// 0 <= L < 2^sh: with H' = H - 2^(52 - sh), which the constant 1.5 2^52 turns into a double,
// fma(H', 2^sh, 2^52 + L) is that sum rounded once (2^52 + L is L's bits under an exponent).
// The power of two is added to the exponent. False (very large inner sizes, results
// outside the normal range): scaled_sum.
__device__ __forceinline__ bool quick_sum(long long hi, int sh, long long lo, double two_sh, int e, double &r) {
  long long h = hi;
  double low = 0.0;
  if (sh) {
    h += (lo >> sh) - (1ll << (52 - sh));
    low = __longlong_as_double((lo & ((1ll << sh) - 1)) | 0x4330000000000000ll);
  }
  bool ok = (unsigned long long)(h + (1ll << 51)) < (1ull << 52);
  double t = __longlong_as_double(h + 0x4338000000000000ll) - 6755399441055744.0;
  if (sh) t = fma(t, two_sh, low);
  const int top = __double2hiint(t), f = (top >> 20) & 0x7ff;
  ok = ok && (f == 0 || (f + e >= 1 && f + e <= 2046));
  r = f ? __hiloint2double(top + e * (1 << 20), __double2loint(t)) : 0.0;
  return ok;
}

// eight columns of an accumulator into registers, and the wait that makes them readable (the
// registers pass through it, so that no use moves before it); with 16 the sums' registers spill
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t (&v)[8]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7])
               : "r"(taddr));
}
__device__ __forceinline__ void tmem_wait8(uint32_t (&v)[8]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+r"(v[0]), "+r"(v[1]), "+r"(v[2]), "+r"(v[3]), "+r"(v[4]), "+r"(v[5]), "+r"(v[6]), "+r"(v[7])
               :
               : "memory");
}

// bounded wait that looks at the barrier before it reads the clock and the limit
__device__ __forceinline__ bool sl_wait(uint32_t bar, uint32_t parity, volatile int *abort_flag) {
  return mbar_try(bar, parity) || mbar_wait(bar, parity, abort_flag);
}

template <int BN>
__global__ void __launch_bounds__(320, 1) k_sl_gemm(const __grid_constant__ SlArgs a) {
  using L = SlTile<BN>;
  extern __shared__ uint8_t smem_raw[];
  uint8_t *smem = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint64_t *full = (uint64_t *)(smem + L::BAR_OFF);
  uint64_t *empty = full + L::ST;
  uint64_t *accf = empty + L::ST;  // a run's accumulators are complete (MMA -> draining warps)
  uint64_t *acce = accf + 1;       // accumulator d drained (draining warps -> MMA)
  uint64_t *fin = acce + 4;
  uint32_t *tmem_slot = (uint32_t *)(fin + 1);
  volatile int *abort_flag = (volatile int *)(tmem_slot + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int s = 0; s < L::ST; ++s) {
      mbar_init(smem_u32(&full[s]), 1);
      mbar_init(smem_u32(&empty[s]), 1);
    }
    mbar_init(smem_u32(accf), 1);
    for (int d = 0; d < 4; ++d) mbar_init(smem_u32(&acce[d]), 4 * L::H);
    mbar_init(smem_u32(fin), 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(L::TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = *tmem_slot;

  if (warp == 0 && lane == 0) {
    // ---------------- TMA producer
    int s = 0, issued = 0, last_s = 0;
    uint32_t par = 1;  // parity of the wait on empty[s]: the first round finds it free
    bool stop = false;
    for (int it = blockIdx.x; it < a.items && !stop; it += gridDim.x) {
      const SlItem d = sl_item<BN>(a, it);
      for (int hi = a.ns + 1; hi >= 2 && !stop; hi -= 4) {
        for (int kb = d.kb_beg; kb < d.kb_end && !stop; ++kb) {
          for (int i = 1; i < hi; ++i) {
            if (!sl_wait(smem_u32(&empty[s]), par, abort_flag)) {
              if (!*abort_flag) *(volatile int *)a.err = 21;
              *abort_flag = 1;
              stop = true;
              break;
            }
            const uint32_t fb = smem_u32(&full[s]);
            mbar_expect_tx(fb, L::STAGE);
            uint8_t *sa = smem + s * L::STAGE;
            tma_load_3d(smem_u32(sa), &a.mA, kb * 64, d.m0, i - 1, fb);
            tma_load_3d(smem_u32(sa + L::ABYTES), &a.mB, kb * 64, d.n0, hi - i - 1, fb);
            ++issued;
            last_s = s;
            if (++s == L::ST) { s = 0; par ^= 1; }
          }
        }
      }
    }
    if (*abort_flag) {
      // drain this CTA's copies in flight before shared memory is released: the
      // last min(issued, ST) loads, each the (issued / ST)-th or so use of its stage
      const int n = issued < L::ST ? issued : L::ST;
      for (int j = 0; j < n; ++j) {
        const int q = issued - 1 - j;  // global index of a load; its stage and use
        int st = last_s - j;
        if (st < 0) st += L::ST;
        mbar_drain(smem_u32(&full[st]), (q / L::ST) & 1);
      }
    }
  } else if (warp == 1) {
    // ---------------- MMA issuer: the warp walks the schedule as one (so that descriptors
    // stay in uniform registers), one elected lane issues
    constexpr uint32_t idesc = idesc_bf16(128, BN);
    const bool lead = elect_one();
    const uint32_t smem0 = __shfl_sync(0xffffffffu, smem_u32(smem), 0);
    const uint32_t acc0 = __shfl_sync(0xffffffffu, tmem, 0);
    const uint32_t desc0 = sdesc_lo(smem0);
    int s = 0;
    uint32_t par = 0, used = 0, epar = 0;  // used, epar: bit d: accumulator d was used, parity of its next wait
    bool stop = false;
    for (int it = blockIdx.x; it < a.items && !stop; it += gridDim.x) {
      const SlItem d = sl_item<BN>(a, it);
      for (int hi = a.ns + 1; hi >= 2 && !stop; hi -= 4) {
        const int nd = pass_classes(hi), run = pass_run(hi, a.b);
        for (int kb0 = d.kb_beg; kb0 < d.kb_end && !stop; kb0 += run) {
          const int kb1 = min(d.kb_end, kb0 + run);
          for (int kb = kb0; kb < kb1 && !stop; ++kb) {
            for (int i = 1; i < hi; ++i) {
              bool ok = sl_wait(smem_u32(&full[s]), par, abort_flag);
              const int dn = min(nd, i);
              const bool fresh = kb == kb0 && i <= nd;  // the first product into accumulator i - 1 of this run
              if (ok && fresh && ((used >> (i - 1)) & 1u)) {
                ok = sl_wait(smem_u32(&acce[i - 1]), (epar >> (i - 1)) & 1u, abort_flag);
                epar ^= 1u << (i - 1);
              }
              if (!__all_sync(0xffffffffu, ok)) {
                if (lane == 0) {
                  if (!*abort_flag) *(volatile int *)a.err = 22;
                  *abort_flag = 1;
                }
                stop = true;
                break;
              }
              fence_after();
              const uint32_t db = desc0 + (uint32_t)((s * L::STAGE + L::ABYTES) >> 4);
              if (lead) {
#pragma unroll
                for (int dd = 0; dd < 4; ++dd) {
                  if (dd >= dn) break;
                  const int sa = s - dd + (s < dd ? L::ST : 0);
                  const uint32_t da = desc0 + (uint32_t)((sa * L::STAGE) >> 4);
                  const uint32_t acc = acc0 + (uint32_t)(dd * BN);
                  const uint32_t keep = (fresh && dd == i - 1) ? 0u : 1u;
                  mma_bf16_lo(acc, da, db, idesc, keep);
#pragma unroll
                  for (int k = 1; k < 4; ++k) mma_bf16_lo(acc, da + 2 * k, db + 2 * k, idesc, 1u);
                }
                // digit i - nd + 1 of A has met its last partner; at the end of the block all have
                if (i >= nd) mma_commit(smem_u32(&empty[s - (nd - 1) + (s < nd - 1 ? L::ST : 0)]));
                if (i == hi - 1)
                  for (int e = nd - 2; e >= 0; --e) mma_commit(smem_u32(&empty[s - e + (s < e ? L::ST : 0)]));
              }
              __syncwarp();
              if (fresh) used |= 1u << (i - 1);
              if (++s == L::ST) { s = 0; par ^= 1; }
            }
          }
          if (!stop && lead) mma_commit(smem_u32(accf));
          __syncwarp();
        }
      }
    }
    // every MMA this warp issued has finished before TMEM is freed
    if (lead) mma_commit(smem_u32(fin));
    __syncwarp();
    mbar_drain(smem_u32(fin), 0);
  } else if (warp >= 2 && warp < 2 + 4 * L::H) {
    // ---------------- draining warps
    const int q = warp & 3, half = (warp - 2) >> 2;
    const int tid = (warp - 2) * 32 + lane;
    constexpr int NT = 128 * L::H;
    const uint32_t tbase = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(half * L::VALS);
    long long *sp = a.spill + (int64_t)blockIdx.x * L::VALS * NT + tid;
    uint32_t par = 0;
    bool ok = true;
    for (int it = blockIdx.x; it < a.items; it += gridDim.x) {
      const SlItem d = sl_item<BN>(a, it);
      long long acc[L::VALS];
      int sh = 0;  // the pass's weight against the first one's: 4 b bits per pass
      for (int hi = a.ns + 1; hi >= 2 && ok; hi -= 4) {
        const int nd = pass_classes(hi), run = pass_run(hi, a.b);
#pragma unroll
        for (int j = 0; j < L::VALS; ++j) acc[j] = 0;
        for (int kb0 = d.kb_beg; kb0 < d.kb_end; kb0 += run) {
          ok = __all_sync(0xffffffffu, sl_wait(smem_u32(accf), par, abort_flag));
          if (!ok) {
            if (lane == 0 && !*abort_flag) { *(volatile int *)a.err = 23; *abort_flag = 1; }
            break;
          }
          par ^= 1;
          fence_after();
          // the next eight columns load while the current ones are added; an accumulator is
          // handed back as soon as its last columns are in registers
          constexpr int CH = L::VALS / 8;
          uint32_t v[2][8];
          tmem_ld8(tbase, v[0]);
          for (int dd = 0; dd < nd; ++dd) {
            const int w = 1 << (a.b * dd);
#pragma unroll
            for (int c = 0; c < CH; ++c) {
              tmem_wait8(v[c & 1]);
              if (c + 1 < CH) {
                tmem_ld8(tbase + (uint32_t)(dd * BN + 8 * (c + 1)), v[(c + 1) & 1]);
              } else {
                fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&acce[dd]));
                if (dd + 1 < nd) tmem_ld8(tbase + (uint32_t)((dd + 1) * BN), v[0]);
              }
#pragma unroll
              for (int j = 0; j < 8; ++j) acc[8 * c + j] += (long long)__float2int_rn(__uint_as_float(v[c & 1][j])) * w;
            }
          }
        }
        if (ok && hi > 5) {  // another pass follows: the sums so far, in units of the first pass, wait
          if (sh == 0) {
#pragma unroll
            for (int j = 0; j < L::VALS; ++j) sp[(int64_t)j * NT] = acc[j];
          } else {
#pragma unroll
            for (int j = 0; j < L::VALS; ++j) sp[(int64_t)j * NT] += acc[j] << sh;
          }
          sh += 4 * a.b;
        }
      }
      // ---- results, in units of 2^(-b (ns + 1))
      const int64_t m = (int64_t)d.m0 + q * 32 + lane;
      if (m >= a.M) continue;
      const unsigned wa = a.WA[m];
      const int n_beg = (d.n0 + half * L::VALS) >> 1;
      const int Nc = a.N2 >> 1;
      // The next column's spilled sums and scale load while the current one is formed (the
      // sums' registers leave no room for more). Four columns per round, the sums moved
      // down in between: unrolled over all of them the code outgrew the instruction cache
      int nh = n_beg / a.n_in, nl = n_beg - nh * a.n_in;
      long long lr = 0, li = 0;
      unsigned wb = a.WB[min(n_beg, Nc - 1)];
      const double two_sh = __hiloint2double((sh + 1023) << 20, 0);
      if (sh) { lr = sp[0]; li = sp[NT]; }
#pragma unroll 1
      for (int j0 = 0; j0 < L::VALS / 2; j0 += 4) {
#pragma unroll
        for (int jj = 0; jj < 4; ++jj) {
          const int n = n_beg + j0 + jj;
          const long long cr = lr, ci = li;
          const unsigned cw = wb;
          const int next = min(j0 + jj + 1, L::VALS / 2 - 1);
          wb = a.WB[min(n_beg + next, Nc - 1)];
          if (sh) { lr = sp[(int64_t)(2 * next) * NT]; li = sp[(int64_t)(2 * next + 1) * NT]; }
          if (n < Nc) {
            cplx val;
            if (!ok || not_finite(wa) || not_finite(cw)) {
              // (after a wait that gave up the tile holds no result)
              val = cmake(__longlong_as_double(0x7ff8000000000000ll), __longlong_as_double(0x7ff8000000000000ll));
            } else {
              const int e = scale_exp(wa) + scale_exp(cw) - a.b * (a.ns + 1);
              const bool qr = quick_sum(acc[2 * jj], sh, cr, two_sh, e, val.x);
              const bool qi = quick_sum(acc[2 * jj + 1], sh, ci, two_sh, e, val.y);
              if (!(qr && qi)) val = cmake(scaled_sum(acc[2 * jj], sh, cr, e), scaled_sum(acc[2 * jj + 1], sh, ci, e));
            }
            if (a.part) {
              a.part[((int64_t)d.split * a.M + m) * Nc + n] = val;
            } else {
              cplx *dst = a.out + m * a.s_m + nh * a.s_nh + nl * a.s_nl;
              if (a.amode == 1) val = cscale(val, a.alpha.x);
              else if (a.amode == 2) val = cmul(a.alpha, val);
              if (a.bmode == 1) { const cplx o = *dst; val = cmake(val.x + a.beta.x * o.x, val.y + a.beta.x * o.y); }
              else if (a.bmode == 2) val = cadd(val, cmul(a.beta, *dst));
              *dst = val;
            }
          }
          if (++nl == a.n_in) { nl = 0; ++nh; }
        }
#pragma unroll
        for (int i = 0; i + 8 < L::VALS; ++i) acc[i] = acc[i + 8];
      }
    }
  }
  fence_before();
  __syncthreads();
  if (warp == 1) {
    __syncwarp();
    fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(L::TMEM_COLS) : "memory");
  }
}

// out = alpha sum_s part[s] + beta out, the splits in order
__global__ void k_sl_reduce(const cplx *__restrict__ part, int ksplit, int64_t M, int64_t Nc, cplx *out, int64_t s_m,
                            int64_t s_nh, int64_t s_nl, int64_t n_in, cplx alpha, int ka, cplx beta, int kb) {
  const int64_t total = M * Nc;
  for (int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; idx < total;
       idx += (int64_t)gridDim.x * blockDim.x) {
    const int64_t m = idx / Nc, n = idx - m * Nc;
    cplx v = cmake(0.0, 0.0);
#pragma unroll 8
    for (int s = 0; s < ksplit; ++s) v = cadd(v, part[(int64_t)s * total + idx]);
    const int64_t nh = n / n_in, nl = n - nh * n_in;
    cplx *dst = out + m * s_m + nh * s_nh + nl * s_nl;
    *dst = axpby(ka, alpha, v, kb, beta, dst);
  }
}

void alloc_sl(Exec &ex, SlMat &d, int64_t rows, int64_t nscale) {
  const size_t bytes = (size_t)d.ns * rows * 2 * d.kp * sizeof(__nv_bfloat16);
  if (d.planes.bytes < bytes) {
    d.planes.reset();
    d.planes = DBuf(ex, bytes);
  }
  if (d.exps.bytes < (size_t)nscale * sizeof(unsigned)) {
    d.exps.reset();
    d.exps = DBuf(ex, (size_t)std::max<int64_t>(nscale, 1) * sizeof(unsigned));
  }
  d.rows = rows;
}

// scales and digits of `rows` complex rows (emb 1: A rows, 2: B rows; cut_from: see sl_pack_A)
void pack_rows(Exec &ex, SlMat &d, const BSrc &s, int64_t rows, int64_t K, bool conj, int emb, int cut_from = 0) {
  alloc_sl(ex, d, emb * rows, rows);
  if (rows <= 0) return;
  ADC_REQUIRE(s.mode == 0 || K < (1ll << 31), ADC_ERR_UNSUPPORTED, "sliced product: ring size");
  const int kfast = pk_kfast(s);
  const int64_t rt = (rows + PK_R - 1) / PK_R;
  const unsigned gx = (unsigned)std::min<int64_t>(rt, 1 << 20);
  unsigned *W = (unsigned *)d.exps.p;
  fill_zero(ex, W, rows * sizeof(unsigned));
  // inner ranges: enough blocks to fill the GPU (a step of 64 elements takes a few
  // microseconds whatever its neighbours do: 16 blocks over 500 elements took 31 us)
  const int64_t want = 8ll * device_sm_count();
  const int64_t parts = std::max<int64_t>(1, std::min<int64_t>((K + PK_K - 1) / PK_K, (want + rt - 1) / rt));
  int64_t krange = (std::max<int64_t>(K, 1) + parts - 1) / parts;
  krange = (krange + PK_K - 1) / PK_K * PK_K;
  const unsigned gy = (unsigned)((std::max<int64_t>(K, 1) + krange - 1) / krange);
  int pr = ex.prof_begin("sl_pack", 0.0, (double)rows * (16.0 * K + 4.0 * emb * d.ns * d.kp));
  k_sl_scale<<<dim3(gx, gy), 256, 0, ex.stream>>>(s, rows, K, krange, kfast, W);
  ADC_CHECK_LAUNCH();
  const dim3 grid(gx, (unsigned)std::min<int64_t>(d.kp / PK_K, 65535));
  const int bits = std::max(d.b * d.ns, cut_from);
  const int64_t pe = (int64_t)emb * rows * 2 * d.kp;
  if (emb == 1)
    k_sl_pack<1><<<grid, 256, 0, ex.stream>>>(s, rows, K, conj ? 1 : 0, d.kp, kfast, W, d.b, d.ns, bits,
                                              (__nv_bfloat16 *)d.planes.p, pe);
  else
    k_sl_pack<2><<<grid, 256, 0, ex.stream>>>(s, rows, K, conj ? 1 : 0, d.kp, kfast, W, d.b, d.ns, bits,
                                              (__nv_bfloat16 *)d.planes.p, pe);
  ADC_CHECK_LAUNCH();
  ex.prof_end(pr);
}

// spill of one CTA with the widest tile
constexpr size_t kSpillCta = (size_t)SlTile<128>::VALS * 128 * SlTile<128>::H * sizeof(long long);

template <int BN>
void launch_sl(Exec &ex, SlArgs &g, SlWork &w, int grid) {
  using L = SlTile<BN>;
  set_smem_limit((const void *)k_sl_gemm<BN>, L::SMEM);
  const size_t need = (size_t)grid * L::VALS * 128 * L::H * sizeof(long long);  // at most kSpillCta per CTA
  if (g.ns > 4 && w.spill.bytes < need) {
    w.spill.reset();
    w.spill = DBuf(ex, need);
  }
  g.spill = (long long *)w.spill.p;
  k_sl_gemm<BN><<<grid, 320, L::SMEM, ex.stream>>>(g);
  ADC_CHECK_LAUNCH();
}

}  // namespace

void sl_set_wait_ns(unsigned long long ns) { ADC_CUDA(cudaMemcpyToSymbol(g_wait_ns, &ns, sizeof(ns))); }

void sl_pack_A(Exec &ex, SlMat &dst, const cplx *src, int64_t M, int64_t K, int64_t s_m, int64_t s_k, bool conj,
               int bits, int cut_from) {
  const SlDigits dg = sl_digits(K, bits);
  dst.kp = sl_kp(K);
  dst.kreal = K;
  dst.b = dg.b;
  dst.ns = dg.ns;
  const BSrc s{src, 0, 0, s_m, std::max<int64_t>(M, 1), s_k, 0, 0, 0, 0};
  pack_rows(ex, dst, s, M, K, conj, 1, cut_from);
}

static void sl_pack_B_impl(Exec &ex, SlMat &dst, const BSrc &s, int64_t Nc, int64_t K, bool conj, const SlMat &like,
                           int bits) {
  ADC_REQUIRE(like.kreal == K, ADC_ERR_ARG, "sl_pack_B: inner size differs from the A operand");
  dst.kp = like.kp;
  dst.kreal = K;
  // fewer significant bits: the leading digits (the product then runs over the
  // common leading slices of both operands)
  dst.b = like.b;
  dst.ns = bits > 0 ? std::min(like.ns, (bits + like.b - 1) / like.b) : like.ns;
  pack_rows(ex, dst, s, Nc, K, conj, 2);
}

void sl_pack_B(Exec &ex, SlMat &dst, const cplx *src, int64_t Nc, int64_t K, int64_t s_nh, int64_t s_nl,
               int64_t n_in, int64_t s_k, bool conj, const SlMat &like, int bits) {
  BSrc s{src, 0, s_nh, s_nl, n_in, s_k, 0, 0, 0, 0};
  // one row index: strides as an A operand, so that the packing sees which index is contiguous
  if (n_in == 1) { s.n_in = std::max<int64_t>(Nc, 1); s.s_nl = s_nh; s.s_nh = 0; }
  sl_pack_B_impl(ex, dst, s, Nc, K, conj, like, bits);
}

void sl_pack_B_ring(Exec &ex, SlMat &dst, const adc_ctx *c, const cplx *X, int64_t k, const SlMat &like, int bits) {
  BSrc s{X, c->kind == ADC_EA ? 1 : 2, 0, 0, 1, 0, c->o, c->v, c->N, c->n1};
  const int64_t Nc = (c->kind == ADC_EA) ? k * c->v : k * c->o;
  sl_pack_B_impl(ex, dst, s, Nc, c->o * c->v, false, like, bits);
}

// a product within Exec::digit_limit: two operand chunks of three eighths, a quarter of
// partial sums, and the spill
constexpr int64_t kDigitLimitMin = (int64_t)64 << 20;
static size_t digit_share(Exec &ex, double part) {
  return (size_t)std::max(0.0, part * ((double)ex.digit_limit - (double)kSpillCta * device_sm_count()));
}

// Tile width and inner split of a product: the ones that leave the SM with the most
// work the least of it, in units of an inner block of a 128-column tile (ns (ns + 1) / 2
// block products of 256 clocks). A 64-column block takes 0.75 and a 32-column one 0.6
// of that (the A operand's reads bound them); a tile's fill, drains and results cost
// about 28 k, 16 k and 16 k clocks; a split costs its partial products, about 10 us
// with the summing kernel's launch.
struct SlPlan {
  int bn = 128, ksplit = 1;
  double clocks = 0.0;
};
constexpr size_t kMaxPartBytes = (size_t)1 << 30;
static SlPlan sl_plan(int64_t M, int64_t N, int64_t kps, int ns, size_t max_part = kMaxPartBytes) {
  const double sms = device_sm_count(), block = 128.0 * ns * (ns + 1);
  const int64_t N2 = 2 * N, tm = (M + 127) / 128;
  SlPlan best;
  best.clocks = 1e300;
  for (int bn = 128; bn >= 32; bn /= 2) {
    if (bn > 32 && bn / 2 >= N2) continue;  // a narrower tile holds every column
    const int64_t tiles = tm * ((N2 + bn - 1) / bn);
    const double per = block * (bn == 128 ? 1.0 : bn == 64 ? 0.75 : 0.6), fixed = bn == 128 ? 28e3 : 16e3;
    for (int s = 1; s <= 64 && (s == 1 || kps / s >= 2); ++s) {
      if (s > 1 && (double)s * M * N * sizeof(cplx) > (double)max_part) break;
      const double red = s > 1 ? 2e4 + (double)(s + 1) * M * N * 0.01 : 0.0;
      const double c = std::ceil(tiles * s / sms) * ((double)((kps + s - 1) / s) * per + fixed) + red;
      if (c < best.clocks) { best.clocks = c; best.bn = bn; best.ksplit = s; }
    }
  }
  return best;
}

void sl_gemm(Exec &ex, const SlMat &A, const SlMat &B, int64_t M, int64_t N, cplx alpha, cplx beta, cplx *out,
             int64_t s_m, int64_t s_nh, int64_t s_nl, int64_t n_in, int *err, SlWork &w) {
  ADC_REQUIRE(A.kp == B.kp && A.b == B.b, ADC_ERR_ARG, "sl_gemm: operands sliced differently");
  ADC_REQUIRE(A.rows >= M && B.rows >= 2 * N, ADC_ERR_ARG, "sl_gemm: operand rows");
  if (M <= 0 || N <= 0) return;
  ADC_REQUIRE(M < (1ll << 31) && 2 * N < (1ll << 31), ADC_ERR_UNSUPPORTED, "sl_gemm: size");
  if (n_in <= 0) n_in = 1;
  const int sms = device_sm_count();
  SlArgs g{};
  g.b = A.b;
  g.ns = std::min(A.ns, B.ns);  // the common leading slices
  const int64_t N2 = 2 * N, kp2 = 2 * A.kp;
  const SlPlan plan = sl_plan(M, N, kp2 / 64, g.ns,
                              ex.digit_limit > 0 ? std::min(kMaxPartBytes, digit_share(ex, 0.25)) : kMaxPartBytes);
  const int bn = plan.bn;
  tc_make_map3(&g.mA, A.planes.p, A.rows, kp2, A.ns, A.rows * kp2, 128);
  tc_make_map3(&g.mB, B.planes.p, B.rows, kp2, B.ns, B.rows * kp2, bn);
  g.M = (int)M;
  g.N2 = (int)N2;
  g.kps = (int)(kp2 / 64);
  g.tiles_m = (int)((M + 127) / 128);
  g.tiles_n = (int)((N2 + bn - 1) / bn);
  g.panel = std::min(g.tiles_n, 8);
  g.WA = (const unsigned *)A.exps.p;
  g.WB = (const unsigned *)B.exps.p;
  g.out = out;
  g.s_m = s_m; g.s_nh = s_nh; g.s_nl = s_nl;
  // one column group covers every column when n_in reaches past them
  g.n_in = (int)std::min<int64_t>(n_in, N);
  g.alpha = alpha;
  g.beta = beta;
  g.amode = alpha.y != 0.0 ? 2 : alpha.x != 1.0 ? 1 : 0;
  g.bmode = beta.y != 0.0 ? 2 : beta.x != 0.0 ? 1 : 0;
  g.err = err;
  const int64_t tiles = (int64_t)g.tiles_m * g.tiles_n;
  g.kb_per_split = (g.kps + plan.ksplit - 1) / plan.ksplit;
  g.ksplit = (g.kps + g.kb_per_split - 1) / g.kb_per_split;
  ADC_REQUIRE(tiles * g.ksplit < (1ll << 31), ADC_ERR_UNSUPPORTED, "sl_gemm: too many tiles");
  g.items = (int)(tiles * g.ksplit);
  if (g.ksplit > 1) {
    const size_t need = (size_t)g.ksplit * M * N * sizeof(cplx);
    if (w.part.bytes < need) {
      w.part.reset();
      const OptionalAlloc opt(ex);
      try {
        w.part = DBuf(ex, need);
      } catch (const Error &e) {
        if (e.code != ADC_ERR_OOM) throw;
        g.ksplit = 1;  // no room for partial products: whole inner sums
        g.kb_per_split = g.kps;
        g.items = (int)tiles;
      }
    }
    if (g.ksplit > 1) g.part = w.part.c();
  }
  const int grid = (int)std::min<int64_t>(g.items, sms);
  // the sliced products count their digit pairs as work, the FP64 ones the product they stand for
  const double flops = 8.0 * (double)M * (double)N * (double)A.kreal;
  const bool fp64 = g.ns * g.b >= kDigitFp64Bits;
  int pr = ex.prof_begin(fp64 ? "tc_digits_fp64" : "tc_sliced_pairs", fp64 ? flops : flops * g.ns * (g.ns + 1) / 2);
  if (bn == 32) launch_sl<32>(ex, g, w, grid);
  else if (bn == 64) launch_sl<64>(ex, g, w, grid);
  else launch_sl<128>(ex, g, w, grid);
  if (g.ksplit > 1) {
    k_sl_reduce<<<grid1d(M * N, 256), 256, 0, ex.stream>>>(g.part, g.ksplit, M, N, out, s_m, s_nh, s_nl, g.n_in,
                                                           alpha, factor_kind(alpha), beta, factor_kind(beta));
    ADC_CHECK_LAUNCH();
  }
  ex.prof_end(pr);
}

// ---------------------------------------------------------------- zgemm through the digits
// > 0: fixed bytes per operand chunk of zgemm_sliced instead of the free-memory rule (test hook)
static size_t g_sliced_cap = 0;
void set_sliced_cap_bytes(size_t bytes) { g_sliced_cap = bytes; }

namespace {

// One batch entry (or a batch folded into the column index: columns n of B at
// (n / n_in) sBh + (n % n_in) sBn, of C at (n / n_in) sCh + (n % n_in) sCn) in
// chunks. The digit planes take 4 ns kp bytes per row of A and 8 ns kp per
// column of B (ns slices of the real embedding): rows and columns in chunks
// whose planes stay within `cap` bytes per operand, so that B is sliced once
// where it fits. When even one 128-row tile of A or 64 columns of B would
// exceed that, the inner index is split as well: the partial products (each
// FP64-accurate) add up in the output. `begun` is set once C may have changed.
void digit_product(Exec &ex, int64_t M, int64_t N, int64_t K, cplx alpha, const cplx *A, int64_t sAm, int64_t sAk,
                   bool conjA, const cplx *B, int64_t sBk, int64_t sBh, int64_t sBn, int64_t n_in, bool conjB,
                   cplx beta, cplx *C, int64_t sCm, int64_t sCh, int64_t sCn, int bits, size_t cap, int *err,
                   SlMat &Sa, SlMat &Sb, SlWork &w, bool &begun) {
  const size_t ns = (size_t)sl_digits(K, bits).ns;
  int64_t kc = K;
  {
    const size_t per = 4 * ns * (size_t)sl_kp(K) * 128;  // one A row tile (B: 64 columns, the same bytes)
    if (per > cap) kc = std::max<int64_t>(512, (int64_t)((double)K * (double)cap / (double)per) / 64 * 64);
  }
  for (int64_t k0 = 0; k0 < K; k0 += kc) {
    const int64_t kk = std::min(kc, K - k0);
    const cplx beta_k = (k0 == 0) ? beta : C1();
    const size_t kp = (size_t)sl_kp(kk), ns = (size_t)sl_digits(kk, bits).ns;
    const int64_t mc = std::min<int64_t>(M, std::max<int64_t>(128, (int64_t)(cap / (4 * ns * kp))));
    int64_t nc = std::min<int64_t>(N, std::max<int64_t>(64, (int64_t)(cap / (8 * ns * kp))));
    if (nc < N && n_in < N) nc = std::max<int64_t>(1, nc / n_in) * n_in;  // whole column groups
    // several chunks: what a later one could need more of than the first is there before out changes
    const size_t spill = (size_t)device_sm_count() * kSpillCta;
    if ((kc < K || mc < M || nc < N) && ns > 4 && w.spill.bytes < spill) {
      w.spill.reset();
      w.spill = DBuf(ex, spill);
    }
    for (int64_t m0 = 0; m0 < M; m0 += mc) {
      const int64_t mm = std::min(mc, M - m0);
      sl_pack_A(ex, Sa, A + m0 * sAm + k0 * sAk, mm, kk, sAm, sAk, conjA, bits);
      for (int64_t n0 = 0; n0 < N; n0 += nc) {
        const int64_t nn = std::min(nc, N - n0);
        const int64_t bo = (n_in < N) ? n0 / n_in * sBh : n0 * sBn, co = (n_in < N) ? n0 / n_in * sCh : n0 * sCn;
        // B once per inner chunk when it fits in one chunk
        if (nc < N || m0 == 0) sl_pack_B(ex, Sb, B + bo + k0 * sBk, nn, kk, sBh, sBn, n_in, sBk, conjB, Sa);
        sl_gemm(ex, Sa, Sb, mm, nn, alpha, beta_k, C + m0 * sCm + co, sCm, sCh, sCn, n_in, err, w);
        begun = true;
      }
    }
  }
}

// smallest operand chunk: its inner index is 512 long (digit_product)
constexpr size_t kDigitCapMin = (size_t)2 << 20;

// Bytes per operand chunk: an eighth of the free device memory, between 1 and 16 GiB (need:
// the larger operand's planes; the free memory is looked up only when they exceed 1 GiB),
// and no more than a third of what the context's limit leaves or its share
size_t digit_cap(Exec &ex, double need) {
  if (g_sliced_cap) return g_sliced_cap;
  size_t cap = (size_t)1 << 30;
  if (need > (double)cap) cap = std::min<size_t>((size_t)16 << 30, std::max(cap, unused_device_memory() / 8));
  if (ex.mem_limit > 0) cap = std::min(cap, (size_t)std::max<int64_t>(0, ex.mem_limit - ex.mem_used) / 3);
  if (ex.digit_limit > 0) cap = std::min(cap, digit_share(ex, 3.0 / 8));
  return std::max(cap, kDigitCapMin);
}

// operand chunks of a product: bytes allowed (0: by digit_cap), bytes of its whole planes
struct DigitChunks {
  size_t cap = 0, whole = 0;
};

// zgemm's operands and output (element strides, conj flags, batch). The larger
// of M and N becomes the A side (half the bytes per digit); a batch whose A
// (or, with the roles exchanged, B) is shared becomes a longer column index.
void digit_zgemm(Exec &ex, int64_t M, int64_t N, int64_t K, int64_t batch, cplx alpha, const cplx *A, int64_t sAb,
                 int64_t sAm, int64_t sAk, bool conjA, const cplx *B, int64_t sBb, int64_t sBk, int64_t sBn,
                 bool conjB, cplx beta, cplx *C, int64_t sCb, int64_t sCm, int64_t sCn, int bits, int *err,
                 bool &begun, DigitChunks &ch) {
  const bool fold = batch > 1 && (sAb == 0 || sBb == 0);
  if (fold ? sAb != 0 : N > M) {
    std::swap(M, N);
    std::swap(A, B);
    std::swap(sAb, sBb);
    std::swap(sAm, sBn);
    std::swap(sAk, sBk);
    std::swap(conjA, conjB);
    std::swap(sCm, sCn);
  }
  SlMat Sa, Sb;
  SlWork w;
  const double need = 4.0 * sl_digits(K, bits).ns * (double)sl_kp(K) * std::max<double>(M, 2.0 * N * (fold ? batch : 1));
  if (!ch.cap) ch.cap = digit_cap(ex, need);
  ch.whole = (size_t)need;
  const size_t cap = ch.cap;
  if (fold) {
    digit_product(ex, M, N * batch, K, alpha, A, sAm, sAk, conjA, B, sBk, sBb, sBn, N, conjB, beta, C, sCm, sCb, sCn,
                  bits, cap, err, Sa, Sb, w, begun);
    return;
  }
  for (int64_t b = 0; b < batch; ++b)
    digit_product(ex, M, N, K, alpha, A + b * sAb, sAm, sAk, conjA, B + b * sBb, sBk, 0, sBn, N, conjB, beta,
                  C + b * sCb, sCm, 0, sCn, bits, cap, err, Sa, Sb, w, begun);
}

}  // namespace

// zgemm as the sliced product: large contractions when Exec::sliced_bits > 0
void zgemm_sliced(Exec &ex, int64_t M, int64_t N, int64_t K, int64_t batch, cplx alpha, const cplx *A, int64_t sAb,
                  int64_t sAm, int64_t sAk, bool conjA, const cplx *B, int64_t sBb, int64_t sBk, int64_t sBn,
                  bool conjB, cplx beta, cplx *C, int64_t sCb, int64_t sCm, int64_t sCn) {
  DBuf err(ex, sizeof(int));
  fill_zero(ex, err.p, sizeof(int));
  bool begun = false;
  DigitChunks ch;
  digit_zgemm(ex, M, N, K, batch, alpha, A, sAb, sAm, sAk, conjA, B, sBb, sBk, sBn, conjB, beta, C, sCb, sCm, sCn,
              ex.sliced_bits, (int *)err.p, begun, ch);
  tc_sync(ex, (int *)err.p);
}

// FP64 products that leave the FP64 units (1.26 TFLOP/s) for the digits: those whose
// estimated time is shorter there. The digits' estimate is their launches (about 45 us
// with both operands' slicing, 25 us with the larger one's digits at hand), the slicing's
// passes over memory at 3 TB/s and the tensor-core kernel's plan; the FP64 units' is their
// kernel's plan. Measured (GB300, M x N x K, FP64 units / digits, slicing included):
// 256^3 110 / 70 us, 384^3 321 / 82 us, 512^3 756 / 118 us, 200 x 8 x 20000 214 / 224 us,
// 1000 x 1000 x 64 391 / 95 us.
static bool digits_pay(int64_t M, int64_t N, int64_t K, int64_t batch, bool kept) {
  if (8.0 * (double)M * (double)N * (double)K * (double)batch < (double)(1 << 24)) return false;
  const double fp64 = zgemm_fp64_clocks(M, N, K, batch);
  N *= batch;  // a shared operand: the batch becomes a longer column index
  if (N > M && !kept) std::swap(M, N);
  constexpr int ns = kDigitFp64Bits / SL_DIGIT;
  const double kp = (double)sl_kp(K);
  const double bytes = (kept ? 0.0 : (double)M * (32.0 * K + 4.0 * ns * kp)) + (double)N * (32.0 * K + 8.0 * ns * kp);
  const double digits = (kept ? 25.0 : 45.0) * 1920.0 + bytes / 3e12 * 1.92e9 + sl_plan(M, N, 2 * sl_kp(K) / 64, ns).clocks;
  return digits < fp64;
}

// a stream under capture keeps the FP64 units (the digit route allocates and may look up free
// memory), and so does a context with next to no memory for it
static bool digits_ready(Exec &ex) {
  cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
  ADC_CUDA(cudaStreamIsCapturing(ex.stream, &cs));
  if (cs != cudaStreamCaptureStatusNone) return false;
  if (ex.digit_limit && ex.digit_limit < kDigitLimitMin) return false;
  if (!ex.digit_err) {
    ADC_CUDA(cudaHostAlloc((void **)&ex.digit_err, sizeof(int), cudaHostAllocMapped));
    *ex.digit_err = 0;
  }
  return true;
}

bool fp64_digits_usable(Exec &ex, int64_t M, int64_t N, int64_t K) {
  return ex.digits != 0 && digits_pay(M, N, K, 1, true) && digits_ready(ex);
}

bool zgemm_fp64_digits(Exec &ex, int64_t M, int64_t N, int64_t K, int64_t batch, cplx alpha, const cplx *A,
                       int64_t sAb, int64_t sAm, int64_t sAk, bool conjA, const cplx *B, int64_t sBb, int64_t sBk,
                       int64_t sBn, bool conjB, cplx beta, cplx *C, int64_t sCb, int64_t sCm, int64_t sCn) {
  const int64_t grouped = (batch > 1 && (sAb == 0 || sBb == 0)) ? batch : 1;
  if (ex.digits == 0 || K <= 0 || (ex.digits == 1 && !digits_pay(M, N, K, grouped, false)) || !digits_ready(ex)) return false;
  const OptionalAlloc opt(ex);
  bool begun = false;
  for (DigitChunks ch;; ch.cap = std::min(ch.cap, ch.whole) / 4) {
    try {
      digit_zgemm(ex, M, N, K, batch, alpha, A, sAb, sAm, sAk, conjA, B, sBb, sBk, sBn, conjB, beta, C, sCb, sCm, sCn,
                  kDigitFp64Bits, ex.digit_err, begun, ch);
      return true;
    } catch (const Error &e) {
      // no room for the digit planes: smaller chunks, then the FP64 units, which need none
      if (e.code != ADC_ERR_OOM || begun) throw;
      if (std::min(ch.cap, ch.whole) / 4 < kDigitCapMin) return false;
    }
  }
}

}  // namespace adc
