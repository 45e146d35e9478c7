// FP64 complex tensor toolkit (see tensor.cuh).
#include <algorithm>
#include <atomic>
#include <chrono>
#include <cstring>
#include <map>
#include <mutex>
#include <set>
#include <thread>
#include <tuple>

#include "tensor.cuh"
#include "tc_slice.cuh"

namespace adc {

// ------------------------------------------------------------------ memory
// Buffers come from one memory pool of the library per device. While contexts
// exist on the device it keeps up to kPoolKeep of freed memory across
// synchronisations: without that every product gave its scratch (hundreds of MB
// of digit planes and gathered blocks) back at its end and mapped it again at
// the next (6.3 of 35 ms in cudaMallocAsync and about as much in the trimming
// synchronisation for an FP64 EA product at o = 30, v = 150, 8 vectors). The last
// context of the device gives everything back.
namespace {
constexpr uint64_t kPoolKeep = 2ull << 30;
struct DevPool {
  cudaMemPool_t pool = nullptr;
  int contexts = 0;
};
std::mutex g_pool_mu;
std::map<int, DevPool> g_pools;

// the pool of device dev (created on first use); call with g_pool_mu held
DevPool &pool_of(int dev) {
  DevPool &d = g_pools[dev];
  if (!d.pool) {
    cudaMemPoolProps pr;
    std::memset(&pr, 0, sizeof(pr));
    pr.allocType = cudaMemAllocationTypePinned;
    pr.handleTypes = cudaMemHandleTypeNone;
    pr.location.type = cudaMemLocationTypeDevice;
    pr.location.id = dev;
    ADC_CUDA(cudaMemPoolCreate(&d.pool, &pr));
  }
  return d;
}
cudaMemPool_t current_pool() {
  int dev = 0;
  ADC_CUDA(cudaGetDevice(&dev));
  std::lock_guard<std::mutex> lk(g_pool_mu);
  return pool_of(dev).pool;
}
}  // namespace

void pool_retain(int dev) {
  std::lock_guard<std::mutex> lk(g_pool_mu);
  DevPool &d = pool_of(dev);
  if (d.contexts == 0) {
    uint64_t keep = kPoolKeep;
    ADC_CUDA(cudaMemPoolSetAttribute(d.pool, cudaMemPoolAttrReleaseThreshold, &keep));
  }
  ++d.contexts;
}

void pool_release(int dev) {
  std::lock_guard<std::mutex> lk(g_pool_mu);
  auto it = g_pools.find(dev);
  if (it == g_pools.end() || it->second.contexts == 0 || --it->second.contexts > 0) return;
  uint64_t keep = 0;
  cudaMemPoolSetAttribute(it->second.pool, cudaMemPoolAttrReleaseThreshold, &keep);
  cudaMemPoolTrimTo(it->second.pool, 0);
}

static int pool_contexts(int dev) {
  std::lock_guard<std::mutex> lk(g_pool_mu);
  auto it = g_pools.find(dev);
  return it == g_pools.end() ? 0 : it->second.contexts;
}

size_t unused_device_memory() {
  size_t fr = 0, tot = 0;
  ADC_CUDA(cudaMemGetInfo(&fr, &tot));
  uint64_t held = 0, used = 0;
  cudaMemPool_t p = current_pool();
  ADC_CUDA(cudaMemPoolGetAttribute(p, cudaMemPoolAttrReservedMemCurrent, &held));
  ADC_CUDA(cudaMemPoolGetAttribute(p, cudaMemPoolAttrUsedMemCurrent, &used));
  return fr + (size_t)(held > used ? held - used : 0);
}

size_t free_device_memory(const Exec *mine) {
  int dev = 0;
  ADC_CUDA(cudaGetDevice(&dev));
  return unused_device_memory() + kept_by_others(dev, mine);
}

// test hook: a device allocation that would take the library's total past the limit fails
static std::atomic<int64_t> g_alloc_limit{0}, g_alloc_total{0}, g_alloc_peak{0};
void set_alloc_limit(int64_t bytes) { g_alloc_limit = bytes; }
int64_t alloc_total() { return g_alloc_total; }
int64_t alloc_peak_reset() { return g_alloc_peak.exchange(g_alloc_total); }

void *Exec::alloc(size_t bytes) {
  if (bytes == 0) return nullptr;
  auto capturing = [&]() {
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    return cudaStreamIsCapturing(stream, &cs) != cudaSuccess || cs != cudaStreamCaptureStatusNone;
  };
  auto over = [&]() { return mem_limit > 0 && mem_used + (int64_t)bytes > mem_limit; };
  if (over() && give_back && !optional && !capturing()) give_back(give_back_of);
  if (over())
    throw Error(ADC_ERR_OOM, "context memory limit exceeded: need " + std::to_string(bytes) +
                                 " bytes, " + std::to_string(mem_used) + " in use of " +
                                 std::to_string(mem_limit));
  void *p = nullptr;
  cudaMemPool_t pool = current_pool();
  auto take = [&]() {
    const int64_t lim = g_alloc_limit;
    return lim > 0 && g_alloc_total + (int64_t)bytes > lim ? cudaErrorMemoryAllocation
                                                           : cudaMallocFromPoolAsync(&p, bytes, pool, stream);
  };
  cudaError_t e = take();
  if (e == cudaErrorMemoryAllocation) {
    // blocks freed on other streams, or kept in sizes that do not fit, go back first
    cudaGetLastError();
    auto again = [&]() {
      if (cudaStreamSynchronize(stream) == cudaSuccess && cudaMemPoolTrimTo(pool, 0) == cudaSuccess)
        e = take();
    };
    if (!capturing()) {
      again();
      // Then what every context of the device keeps for speed. A context inside a product keeps
      // its digits and holds that product's planes until it is enqueued: with others
      // there, look again for a tenth of a second
      int dev = 0;
      const int looks = !optional && cudaGetDevice(&dev) == cudaSuccess ? (pool_contexts(dev) > 1 ? 50 : 1) : 0;
      for (int t = 0; e == cudaErrorMemoryAllocation && t < looks; ++t) {
        if (t) std::this_thread::sleep_for(std::chrono::milliseconds(2));
        cudaGetLastError();
        if (reclaim_kept_digits(dev) || t) again();
      }
    }
  }
  if (e != cudaSuccess) {
    cudaGetLastError();
    throw Error(e == cudaErrorMemoryAllocation ? ADC_ERR_OOM : ADC_ERR_CUDA,
                std::string("cudaMallocFromPoolAsync(") + std::to_string(bytes) + "): " + cudaGetErrorString(e) +
                    " (" + std::to_string(mem_used) + " bytes held by the context" +
                    (stage.empty() ? std::string() : ", in " + stage) + (tag.empty() ? std::string() : "/" + tag) +
                    ")");
  }
  const int64_t now = g_alloc_total += (int64_t)bytes;
  for (int64_t top = g_alloc_peak; now > top && !g_alloc_peak.compare_exchange_weak(top, now);) {
  }
  mem_used += (int64_t)bytes;
  mem_peak = std::max<int64_t>(mem_peak, mem_used);
  return p;
}

void Exec::release(void *p, size_t bytes) {
  if (!p) return;
  cudaFreeAsync(p, stream);
  g_alloc_total -= (int64_t)bytes;
  mem_used -= (int64_t)bytes;
}

long long g_launches = 0;

int Exec::take_digits() {
  if (!digit_err) return 0;
  const int h = *(volatile int *)digit_err;
  *digit_err = 0;
  return h;
}

void Exec::sync() {
  ADC_CUDA(cudaStreamSynchronize(stream));
  check_digits();
}

void Exec::check_digits() {
  const int h = take_digits();
  if (h) throw Error(ADC_ERR_TIMEOUT, "FP64 product: a tensor-core wait gave up (code " + std::to_string(h) + ")");
}

cudaEvent_t Exec::event() {
  if (!event_pool.empty()) {
    cudaEvent_t e = event_pool.back();
    event_pool.pop_back();
    return e;
  }
  cudaEvent_t e;
  ADC_CUDA(cudaEventCreate(&e));
  return e;
}

int Exec::prof_begin(const char *kernel, double flops, double bytes) {
  if (!prof) return -1;
  ProfRec r;
  r.name = std::string(kernel) + (tag.empty() ? "" : "/" + tag);
  r.a = event();
  r.b = event();
  r.flops = flops;
  r.bytes = bytes;
  ADC_CUDA(cudaEventRecord(r.a, stream));
  recs.push_back(r);
  return (int)recs.size() - 1;
}

void Exec::prof_end(int r) {
  if (r >= 0) ADC_CUDA(cudaEventRecord(recs[r].b, stream));
}

void Exec::prof_clear() {
  for (auto &r : recs) {
    event_pool.push_back(r.a);
    event_pool.push_back(r.b);
  }
  recs.clear();
}

void fill_zero(Exec &ex, void *p, size_t bytes) {
  if (bytes) ADC_CUDA(cudaMemsetAsync(p, 0, bytes, ex.stream));
}

// ------------------------------------------------------------------ GEMM
// FP64 units (two multiply-adds a clock and SM on GB300) bound every product
// here, so what counts is to give them no padding and to use every SM: the
// output tile is chosen by shape from 64 x 64 down to strips of four rows or
// columns (the k trial vectors of a product), and the inner index is split
// over CTAs, each CTA's partial tile going to a buffer that the tile's last
// CTA sums in the splits' order. The loads only need to be coalesced along
// whichever operand index has unit stride; K is staged 16 at a time, the next
// stage's elements loaded while the current one is used.
// Measured (GB300, M x N x K, one 64 x 64 tile for every shape before / now): 16^3
// 55 / 6 us, 64^3 63 / 12 us, 128^3 66 / 25 us, 4 x 672 x 8 57 / 6 us, 200 x 8 x 20000
// 1.71 / 0.21 ms, 20000 x 8 x 200 1.94 / 0.22 ms (0.15 at the FP64 units' rate),
// 4 x 1156 x 1156 511 / 59 us, 512^3 0.78 / 0.76 ms (0.64).
namespace {
constexpr int BKK = 16;

struct ZArgs {
  int64_t M, N, K;
  const cplx *A;
  int64_t sAb, sAm, sAk;
  const cplx *B;
  int64_t sBb, sBk, sBn;
  cplx *C;
  int64_t sCb, sCm, sCn;
  cplx alpha, beta;
  int64_t batch0, kchunk, nbatch;
  int conjA, a_kfast, conjB, b_nfast, ksplit, mfast;
  cplx *part;     // [ksplit][nbatch][M][N] partial products (ksplit > 1)
  unsigned *cnt;  // a counter per output tile (zero between launches), or null: k_splitk_reduce follows
};

template <int BM, int BN, int TM, int TN>
__global__ void __launch_bounds__((BM / TM) * (BN / TN)) k_zgemm(const ZArgs z) {
  // 3M products: (ar + i ai)(br + i bi) = T1 - T2 + i (T3 - T1 - T2) with
  // T1 = ar br, T2 = ai bi, T3 = (ar + ai)(br + bi): three FP64 FMAs per
  // complex MAC instead of four. The sums are formed once per staged element.
  constexpr int RM = BM / TM, RN = BN / TN, NT = RM * RN;
  constexpr int LA = (BM * BKK + NT - 1) / NT, LB = (BN * BKK + NT - 1) / NT;
  extern __shared__ double zsm[];
  cplx(*As)[BM + 1] = reinterpret_cast<cplx(*)[BM + 1]>(zsm);
  cplx(*Bs)[BN + 1] = reinterpret_cast<cplx(*)[BN + 1]>(zsm + 2 * BKK * (BM + 1));
  double(*Ass)[BM + 1] = reinterpret_cast<double(*)[BM + 1]>(zsm + 2 * BKK * (BM + 1) + 2 * BKK * (BN + 1));
  double(*Bss)[BN + 1] = reinterpret_cast<double(*)[BN + 1]>(zsm + 3 * BKK * (BM + 1) + 2 * BKK * (BN + 1));
  const int tid = threadIdx.x;
  const int tx = tid % RN, ty = tid / RN;
  const int64_t zl = blockIdx.z;
  const int64_t split = zl % z.ksplit;
  const int64_t bl = zl / z.ksplit;
  const int64_t b = bl + z.batch0;
  // with mfast the row tiles vary fastest, so the CTAs that read one column
  // tile of B (the large operand of the skinny shapes) run together and share it in L2
  const int64_t m0 = (int64_t)(z.mfast ? blockIdx.x : blockIdx.y) * BM;
  const int64_t n0 = (int64_t)(z.mfast ? blockIdx.y : blockIdx.x) * BN;
  const int64_t kbeg = split * z.kchunk;
  const int64_t kend = (kbeg + z.kchunk < z.K) ? kbeg + z.kchunk : z.K;
  const cplx *Ab = z.A + b * z.sAb;
  const cplx *Bb = z.B + b * z.sBb;
  double t1[TM][TN], t2[TM][TN], t3[TM][TN];
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TN; ++j) t1[i][j] = t2[i][j] = t3[i][j] = 0.0;
  const double sa = z.conjA ? -1.0 : 1.0, sb = z.conjB ? -1.0 : 1.0;
  cplx ra[LA], rb[LB];
  auto load = [&](int64_t k0) {
#pragma unroll
    for (int r = 0; r < LA; ++r) {
      const int idx = tid + NT * r;
      const int kk = z.a_kfast ? idx % BKK : idx / BM, mm = z.a_kfast ? idx / BKK : idx % BM;
      const int64_t gm = m0 + mm, gk = k0 + kk;
      ra[r] = (idx < BM * BKK && gm < z.M && gk < kend) ? Ab[gm * z.sAm + gk * z.sAk] : cmake(0.0, 0.0);
    }
#pragma unroll
    for (int r = 0; r < LB; ++r) {
      const int idx = tid + NT * r;
      const int kk = z.b_nfast ? idx / BN : idx % BKK, nn = z.b_nfast ? idx % BN : idx / BKK;
      const int64_t gn = n0 + nn, gk = k0 + kk;
      rb[r] = (idx < BN * BKK && gn < z.N && gk < kend) ? Bb[gk * z.sBk + gn * z.sBn] : cmake(0.0, 0.0);
    }
  };
  load(kbeg);
  for (int64_t k0 = kbeg; k0 < kend; k0 += BKK) {
#pragma unroll
    for (int r = 0; r < LA; ++r) {
      const int idx = tid + NT * r;
      const int kk = z.a_kfast ? idx % BKK : idx / BM, mm = z.a_kfast ? idx / BKK : idx % BM;
      if (BM * BKK % NT != 0 && idx >= BM * BKK) continue;
      const cplx v = cmake(ra[r].x, ra[r].y * sa);
      As[kk][mm] = v;
      Ass[kk][mm] = v.x + v.y;
    }
#pragma unroll
    for (int r = 0; r < LB; ++r) {
      const int idx = tid + NT * r;
      const int kk = z.b_nfast ? idx / BN : idx % BKK, nn = z.b_nfast ? idx % BN : idx / BKK;
      if (BN * BKK % NT != 0 && idx >= BN * BKK) continue;
      const cplx v = cmake(rb[r].x, rb[r].y * sb);
      Bs[kk][nn] = v;
      Bss[kk][nn] = v.x + v.y;
    }
    __syncthreads();
    if (k0 + BKK < kend) load(k0 + BKK);
    // (the last stage holds only the elements there are: the FP64 units do no padding)
    const int kn = (int)(kend - k0 < BKK ? kend - k0 : BKK);
#pragma unroll 4
    for (int kk = 0; kk < kn; ++kk) {
      cplx a[TM], bv[TN];
      double as[TM], bs[TN];
#pragma unroll
      for (int i = 0; i < TM; ++i) { a[i] = As[kk][ty + RM * i]; as[i] = Ass[kk][ty + RM * i]; }
#pragma unroll
      for (int j = 0; j < TN; ++j) { bv[j] = Bs[kk][tx + RN * j]; bs[j] = Bss[kk][tx + RN * j]; }
#pragma unroll
      for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TN; ++j) {
          t1[i][j] = fma(a[i].x, bv[j].x, t1[i][j]);
          t2[i][j] = fma(a[i].y, bv[j].y, t2[i][j]);
          t3[i][j] = fma(as[i], bs[j], t3[i][j]);
        }
    }
    __syncthreads();
  }
  cplx acc[TM][TN];
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TN; ++j) acc[i][j] = cmake(t1[i][j] - t2[i][j], t3[i][j] - t1[i][j] - t2[i][j]);
  if (z.ksplit > 1) {
    // split-K partial tile, unscaled: part[split][bl][m][n]
    const int64_t step = z.nbatch * z.M * z.N;
    cplx *P = z.part + bl * z.M * z.N;
#pragma unroll
    for (int i = 0; i < TM; ++i) {
      const int64_t gm = m0 + ty + RM * i;
#pragma unroll
      for (int j = 0; j < TN; ++j) {
        const int64_t gn = n0 + tx + RN * j;
        if (gm < z.M && gn < z.N) P[split * step + gm * z.N + gn] = acc[i][j];
      }
    }
    if (!z.cnt) return;
    // the CTA that finds every other split's tile written sums them, in order
    __shared__ unsigned seen;
    __threadfence();
    __syncthreads();
    unsigned *cnt = z.cnt + ((int64_t)bl * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x;
    if (tid == 0) seen = atomicAdd(cnt, 1u);
    __syncthreads();
    if (seen != (unsigned)z.ksplit - 1) return;
    __threadfence();
    if (tid == 0) *cnt = 0;
#pragma unroll
    for (int i = 0; i < TM; ++i) {
      const int64_t gm = m0 + ty + RM * i;
#pragma unroll
      for (int j = 0; j < TN; ++j) {
        const int64_t gn = n0 + tx + RN * j;
        cplx s = cmake(0.0, 0.0);
        if (gm < z.M && gn < z.N) {
          const cplx *p = P + gm * z.N + gn;
#pragma unroll 8
          for (int k = 0; k < z.ksplit; ++k) s = cadd(s, __ldcg(p + k * step));
        }
        acc[i][j] = s;
      }
    }
  }
  cplx *Cb = z.C + b * z.sCb;
  const bool use_beta = (z.beta.x != 0.0 || z.beta.y != 0.0);
#pragma unroll
  for (int i = 0; i < TM; ++i) {
    int64_t gm = m0 + ty + RM * i;
    if (gm >= z.M) continue;
#pragma unroll
    for (int j = 0; j < TN; ++j) {
      int64_t gn = n0 + tx + RN * j;
      if (gn >= z.N) continue;
      cplx *dst = Cb + gm * z.sCm + gn * z.sCn;
      cplx r = cmul(z.alpha, acc[i][j]);
      if (use_beta) r = cadd(r, cmul(z.beta, *dst));
      *dst = r;
    }
  }
}
__global__ void k_splitk_reduce(const cplx *__restrict__ part, int ksplit, int64_t nb, int64_t M,
                                int64_t N, cplx *C, int64_t sCb, int64_t sCm, int64_t sCn,
                                cplx alpha, cplx beta, int64_t batch0) {
  const int64_t total = nb * M * N;
  const bool use_beta = (beta.x != 0.0 || beta.y != 0.0);
  for (int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; idx < total;
       idx += (int64_t)gridDim.x * blockDim.x) {
    int64_t n = idx % N, r = idx / N;
    int64_t m = r % M, bl = r / M;
    cplx s = cmake(0.0, 0.0);
    for (int k = 0; k < ksplit; ++k) s = cadd(s, part[(int64_t)k * total + idx]);
    cplx *dst = C + (bl + batch0) * sCb + m * sCm + n * sCn;
    cplx res = cmul(alpha, s);
    if (use_beta) res = cadd(res, cmul(beta, *dst));
    *dst = res;
  }
}
}  // namespace

namespace {
std::mutex g_dev_mu;
std::map<int, int> g_dev_sms;
std::set<std::tuple<const void *, int, int>> g_smem_set;
}  // namespace

int device_sm_count() {
  int dev = 0;
  ADC_CUDA(cudaGetDevice(&dev));
  std::lock_guard<std::mutex> lk(g_dev_mu);
  auto it = g_dev_sms.find(dev);
  if (it != g_dev_sms.end()) return it->second;
  int s = 0;
  ADC_CUDA(cudaDeviceGetAttribute(&s, cudaDevAttrMultiProcessorCount, dev));
  if (s <= 0) s = 148;
  g_dev_sms[dev] = s;
  return s;
}

void set_smem_limit(const void *kernel, int bytes) {
  int dev = 0;
  ADC_CUDA(cudaGetDevice(&dev));
  std::lock_guard<std::mutex> lk(g_dev_mu);
  const auto key = std::make_tuple(kernel, dev, bytes);
  if (g_smem_set.count(key)) return;
  ADC_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes));
  g_smem_set.insert(key);
}

static int num_sms() { return device_sm_count(); }

namespace {
// output tiles of the FP64 kernel
struct ZTile {
  int bm, bn;
  void (*kernel)(const ZArgs);
  int threads;
};
const ZTile kZTiles[] = {
    {64, 64, k_zgemm<64, 64, 4, 4>, 256}, {32, 32, k_zgemm<32, 32, 2, 2>, 256}, {16, 16, k_zgemm<16, 16, 2, 2>, 64},
    {8, 32, k_zgemm<8, 32, 2, 2>, 64},    {32, 8, k_zgemm<32, 8, 2, 2>, 64},    {4, 64, k_zgemm<4, 64, 2, 2>, 64},
    {64, 4, k_zgemm<64, 4, 2, 2>, 64},    {8, 8, k_zgemm<8, 8, 1, 1>, 64}};

// Tile and inner split of the least estimated time, in clocks: the SM with the
// most CTAs runs ceil(CTAs / SMs) tiles at two multiply-adds a clock (three per
// complex one, and the staging adds), half a one per scheduler, so that fewer
// than four warps on an SM leave part of it idle; each stage of a CTA costs a
// load latency that the SM's other CTAs hide; a split's partial sums cost a pass
// through L2 by the tile's last CTA (or a second kernel).
// max_split: 1 without a workspace; the partial products stay within max_part elements.
struct ZPlan {
  const ZTile *t = nullptr;
  int ksplit = 1;
  double clocks = 0.0;
};
ZPlan z_plan(int64_t M, int64_t N, int64_t K, int64_t batch, int max_split, int64_t max_part, bool fused) {
  static const int kSplits[] = {1, 2, 3, 4, 6, 8, 12, 16, 24, 32, 48, 64};
  const double sms = num_sms();
  ZPlan best;
  best.clocks = 1e300;
  for (const ZTile &t : kZTiles) {
    const int64_t tm = (M + t.bm - 1) / t.bm, tn = (N + t.bn - 1) / t.bn;
    if (std::min(tm, tn) > 65535) continue;
    const double tiles = (double)tm * (double)tn * (double)batch;
    for (int s : kSplits) {
      if (s > max_split) break;
      if (s > 1 && (s > (K + BKK - 1) / BKK || (double)s * M * N * batch > (double)max_part)) break;
      const double stages = std::ceil((double)((K + s - 1) / s) / BKK);
      const double per = std::ceil(tiles * s / sms);
      const double kk = std::min<double>(stages * BKK, std::max<double>(K, 1));
      const double work = per * (1.5 * t.bm * t.bn + 0.5 * (t.bm + t.bn)) * kk * std::max(1.0, 4.0 / (per * t.threads / 32));
      const double lat = stages * 1100.0 * std::ceil(per * t.threads / 512.0);
      const double red = s == 1 ? 0.0 : fused ? 2500.0 + 80.0 * s : 8000.0 + 20.0 * s;
      const double c = std::max(work, lat) + 0.3 * std::min(work, lat) + red;
      if (c < best.clocks) { best.clocks = c; best.t = &t; best.ksplit = s; }
      if (tiles * s > 8.0 * sms) break;
    }
  }
  return best;
}

// one FP64 product with the tile and split of p, in batch slices; part: room for
// ksplit partial products of a slice of at most slice(batch) entries; cnt as ZArgs::cnt
void z_launch(Exec &ex, const ZPlan &p, ZArgs z, int64_t batch, cplx *part, unsigned *cnt) {
  const int64_t mt = (z.M + p.t->bm - 1) / p.t->bm, nt = (z.N + p.t->bn - 1) / p.t->bn;
  z.mfast = (nt <= 65535) ? 1 : 0;
  ADC_REQUIRE(z.mfast || mt <= 65535, ADC_ERR_UNSUPPORTED, "zgemm: shape too large");
  z.a_kfast = (z.sAk == 1) ? 1 : 0;
  z.b_nfast = (z.sBn == 1) ? 1 : 0;
  z.ksplit = p.ksplit;
  z.kchunk = (z.K + p.ksplit - 1) / p.ksplit;
  if (p.ksplit > 1) z.kchunk = (z.kchunk + BKK - 1) / BKK * BKK;
  z.part = part;
  z.cnt = cnt;
  const int64_t bmax = 65535 / p.ksplit;
  const int smem = 3 * BKK * (p.t->bm + 1 + p.t->bn + 1) * (int)sizeof(double);
  if (smem > 48 * 1024 - 64) set_smem_limit((const void *)p.t->kernel, smem);
  for (int64_t b0 = 0; b0 < batch; b0 += bmax) {
    z.nbatch = std::min<int64_t>(bmax, batch - b0);
    z.batch0 = b0;
    const dim3 grid(z.mfast ? (unsigned)mt : (unsigned)nt, z.mfast ? (unsigned)nt : (unsigned)mt,
                    (unsigned)(z.nbatch * p.ksplit));
    p.t->kernel<<<grid, p.t->threads, smem, ex.stream>>>(z);
    ADC_CHECK_LAUNCH();
    if (p.ksplit > 1 && !cnt) {
      k_splitk_reduce<<<grid1d(z.nbatch * z.M * z.N, 256), 256, 0, ex.stream>>>(
          part, p.ksplit, z.nbatch, z.M, z.N, z.C, z.sCb, z.sCm, z.sCn, z.alpha, z.beta, b0);
      ADC_CHECK_LAUNCH();
    }
  }
}
constexpr int64_t kMaxPart = (int64_t)1 << 26;  // elements of a call's partial products
}  // namespace

double zgemm_fp64_clocks(int64_t M, int64_t N, int64_t K, int64_t batch) {
  return z_plan(M, N, K, batch, 64, kMaxPart, true).clocks;
}

void zgemm(Exec &ex, int64_t M, int64_t N, int64_t K, int64_t batch, cplx alpha, const cplx *A,
           int64_t sAb, int64_t sAm, int64_t sAk, bool conjA, const cplx *B, int64_t sBb,
           int64_t sBk, int64_t sBn, bool conjB, cplx beta, cplx *C, int64_t sCb, int64_t sCm,
           int64_t sCn) {
  if (M <= 0 || N <= 0 || batch <= 0) return;
  if (K < 0) K = 0;  // the kernel then writes beta * C
  // (short inner sizes stay here: there the product is bound by memory, and the
  // sliced form reads and writes several times more)
  if (ex.sliced_bits > 0 && K >= 512 && 8.0 * (double)M * N * K * batch >= (double)(1 << 24)) {
    ex.n_sliced += 1;
    ex.flops_sliced += 8.0 * (double)M * N * K * batch;
    zgemm_sliced(ex, M, N, K, batch, alpha, A, sAb, sAm, sAk, conjA, B, sBb, sBk, sBn, conjB, beta, C, sCb, sCm,
                 sCn);
    return;
  }
  ex.n_fp64 += 1;
  ex.flops_fp64 += 8.0 * (double)M * N * K * batch;
  if (zgemm_fp64_digits(ex, M, N, K, batch, alpha, A, sAb, sAm, sAk, conjA, B, sBb, sBk, sBn, conjB, beta, C, sCb,
                        sCm, sCn))
    return;
  const ZArgs z{M, N, K, A, sAb, sAm, sAk, B, sBb, sBk, sBn, C, sCb, sCm, sCn, alpha, beta, 0, 0, 0,
                conjA ? 1 : 0, 0, conjB ? 1 : 0, 0, 1, 0, nullptr, nullptr};
  ZPlan p = z_plan(M, N, K, batch, 64, kMaxPart, ex.zcount.p != nullptr);
  ADC_REQUIRE(p.t, ADC_ERR_UNSUPPORTED, "zgemm: shape too large");
  DBuf part;
  unsigned *cnt = nullptr;
  cplx *pp = nullptr;
  if (p.ksplit > 1) {
    const int64_t slice = std::min<int64_t>(batch, 65535 / p.ksplit);
    const int64_t tiles = (M + p.t->bm - 1) / p.t->bm * ((N + p.t->bn - 1) / p.t->bn) * slice;
    if (tiles <= (int64_t)(ex.zcount.bytes / sizeof(unsigned))) cnt = (unsigned *)ex.zcount.p;
    // the partial products: the context's own small buffer, or one of the call
    if (cnt && (size_t)p.ksplit * slice * M * N * sizeof(cplx) <= ex.zpart.bytes) {
      pp = (cplx *)ex.zpart.p;
    } else {
      const OptionalAlloc opt(ex);
      try {
        part = cbuf(ex, (int64_t)p.ksplit * slice * M * N);
        pp = part.c();
      } catch (const Error &e) {  // no room for them: whole inner sums
        if (e.code != ADC_ERR_OOM) throw;
        p = z_plan(M, N, K, batch, 1, 0, false);
        ADC_REQUIRE(p.t, ADC_ERR_UNSUPPORTED, "zgemm: shape too large");
        cnt = nullptr;
      }
    }
  }
  int pr = ex.prof_begin("zgemm_fp64", 8.0 * (double)M * N * K * batch,
                         16.0 * (double)batch * ((double)M * K + (double)K * N + (double)M * N));
  z_launch(ex, p, z, batch, pp, cnt);
  ex.prof_end(pr);
}

void zgemm_ws(Exec &ex, int64_t M, int64_t N, int64_t K, int64_t batch, cplx alpha, const cplx *A,
              int64_t sAb, int64_t sAm, int64_t sAk, bool conjA, const cplx *B, int64_t sBb, int64_t sBk,
              int64_t sBn, bool conjB, cplx beta, cplx *C, int64_t sCb, int64_t sCm, int64_t sCn, cplx *ws,
              int64_t ws_elems) {
  if (M <= 0 || N <= 0 || batch <= 0) return;
  if (K < 0) K = 0;
  const ZArgs z{M, N, K, A, sAb, sAm, sAk, B, sBb, sBk, sBn, C, sCb, sCm, sCn, alpha, beta, 0, 0, 0,
                conjA ? 1 : 0, 0, conjB ? 1 : 0, 0, 1, 0, nullptr, nullptr};
  // the splits are capped by the workspace the caller provides
  const ZPlan p = z_plan(M, N, K, batch, ws ? 64 : 1, ws_elems, false);
  ADC_REQUIRE(p.t, ADC_ERR_UNSUPPORTED, "zgemm: shape too large");
  z_launch(ex, p, z, batch, ws, nullptr);
}

// ------------------------------------------------------------------ permute
namespace {
constexpr int MAXD = 8;
struct PermArgs {
  int nd;
  int strided_dst;  // 0: dst contiguous in ext order; 1: dst at strides dstr
  int64_t ext[MAXD];
  int64_t sstr[MAXD];
  int64_t dstr[MAXD];
  FastDiv fd[MAXD];
};

// (measured on 2.6 M elements of four axes: 36 us with 64-bit divisions and a complex factor)
template <bool SMALL>
__global__ void k_permute(const cplx *__restrict__ src, PermArgs pa, int conj, cplx *dst, cplx alpha, int ka,
                          cplx beta, int kb, int64_t total) {
  for (int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; idx < total;
       idx += (int64_t)gridDim.x * blockDim.x) {
    int64_t off = 0, doff = 0;
    if (SMALL) {  // fewer than 2^31 elements
      uint32_t rem = (uint32_t)idx;
      for (int d = pa.nd - 1; d >= 0; --d) {
        const uint32_t q = fdiv(rem, pa.fd[d]), i = rem - q * pa.fd[d].d;
        rem = q;
        off += i * pa.sstr[d];
        doff += i * pa.dstr[d];
      }
    } else {
      int64_t rem = idx;
      for (int d = pa.nd - 1; d >= 0; --d) {
        int64_t i = rem % pa.ext[d];
        rem /= pa.ext[d];
        off += i * pa.sstr[d];
        doff += i * pa.dstr[d];
      }
    }
    if (!pa.strided_dst) doff = idx;
    cplx v = src[off];
    if (conj) v.y = -v.y;
    dst[doff] = axpby(ka, alpha, v, kb, beta, dst + doff);
  }
}

void launch_permute(Exec &ex, const cplx *src, PermArgs &pa, bool conj, cplx *dst, cplx alpha, cplx beta,
                    int64_t total) {
  const int ka = factor_kind(alpha), kb = factor_kind(beta);
  if (total < (1ll << 31)) {
    for (int d = 0; d < pa.nd; ++d) pa.fd[d] = fast_div((uint32_t)pa.ext[d]);
    k_permute<true><<<grid1d(total, 256), 256, 0, ex.stream>>>(src, pa, conj ? 1 : 0, dst, alpha, ka, beta, kb, total);
  } else {
    k_permute<false><<<grid1d(total, 256), 256, 0, ex.stream>>>(src, pa, conj ? 1 : 0, dst, alpha, ka, beta, kb, total);
  }
  ADC_CHECK_LAUNCH();
}
}  // namespace

void permute(Exec &ex, const cplx *src, const std::vector<int64_t> &ext, const std::vector<int64_t> &sstr,
             bool conj, cplx *dst, const std::vector<int64_t> &dstr, cplx alpha, cplx beta) {
  PermArgs pa{};
  ADC_REQUIRE(ext.size() <= (size_t)MAXD && ext.size() == sstr.size() && ext.size() == dstr.size(), ADC_ERR_ARG,
              "permute: rank");
  pa.nd = (int)ext.size();
  pa.strided_dst = 1;
  int64_t total = 1;
  for (int d = 0; d < pa.nd; ++d) {
    pa.ext[d] = ext[d];
    pa.sstr[d] = sstr[d];
    pa.dstr[d] = dstr[d];
    total *= ext[d];
  }
  if (total == 0) return;
  launch_permute(ex, src, pa, conj, dst, alpha, beta, total);
}

void permute(Exec &ex, const cplx *src, const std::vector<int64_t> &ext,
             const std::vector<int64_t> &sstr, bool conj, cplx *dst, cplx alpha, cplx beta) {
  PermArgs pa{};
  ADC_REQUIRE(ext.size() <= (size_t)MAXD && ext.size() == sstr.size(), ADC_ERR_ARG, "permute: rank");
  pa.nd = (int)ext.size();
  int64_t total = 1;
  for (int d = 0; d < pa.nd; ++d) { pa.ext[d] = ext[d]; pa.sstr[d] = sstr[d]; total *= ext[d]; }
  if (pa.nd == 0) { pa.nd = 1; pa.ext[0] = 1; pa.sstr[0] = 0; }
  if (total == 0) return;
  launch_permute(ex, src, pa, conj, dst, alpha, beta, total);
}

// ------------------------------------------------------------------ pairs
namespace {
__global__ void k_pair_unpack(const cplx *__restrict__ P, int64_t no1, int64_t no0, int64_t sP1,
                              int64_t sP0, int64_t n, int64_t inner, cplx *T, int64_t total) {
  for (int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; idx < total;
       idx += (int64_t)gridDim.x * blockDim.x) {
    int64_t in = idx % inner;
    int64_t r = idx / inner;
    int64_t q = r % n; r /= n;
    int64_t p = r % n; r /= n;
    int64_t o0 = r % no0, o1 = r / no0;
    cplx v = cmake(0.0, 0.0);
    if (p < q) v = P[o1 * sP1 + o0 * sP0 + pair_index(p, q, n) * inner + in];
    else if (p > q) { v = P[o1 * sP1 + o0 * sP0 + pair_index(q, p, n) * inner + in]; v.x = -v.x; v.y = -v.y; }
    T[idx] = v;
  }
}

// The same for inner = 1 and one unit stride of T (sTq == 1, or sTp == 1 when qfast is 0):
// a block takes the 32 x 32 tiles (p, q) and (q, p) of one outer index through shared
// memory, so that T is read along its unit stride and P written along q
__global__ void __launch_bounds__(256)
k_pair_pack_tile(const cplx *__restrict__ T, int64_t sTo1, int64_t sTo0, int64_t ld, int qfast, double s, int64_t no0,
                 int64_t n, cplx *P, int64_t sP1, int64_t sP0, cplx alpha, int ka, cplx beta, int kb) {
  __shared__ cplx a[32][33], b[32][33];  // a[p][q] = T(p0 + p, q0 + q), b[q][p] = T(q0 + q, p0 + p)
  // blockIdx.x counts the tile pairs pb <= qb row by row
  const int nt = (int)((n + 31) / 32);
  int pb = 0, r = blockIdx.x;
  while (r >= nt - pb) { r -= nt - pb; ++pb; }
  const int64_t p0 = 32 * pb, q0 = 32 * (pb + r);
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  const int64_t o0 = blockIdx.y % no0, o1 = blockIdx.y / no0;
  const cplx *Tb = T + o1 * sTo1 + o0 * sTo0;
#pragma unroll
  for (int i = ty; i < 32; i += 8) {
    // rows of memory: qfast: T(p, .) at p ld, else T(., q) at q ld
    const int64_t x = (qfast ? p0 : q0) + i, y = (qfast ? q0 : p0) + tx;
    if (x < n && y < n) (qfast ? a[i][tx] : a[tx][i]) = Tb[x * ld + y];
    const int64_t x2 = (qfast ? q0 : p0) + i, y2 = (qfast ? p0 : q0) + tx;
    if (s != 0.0 && x2 < n && y2 < n) (qfast ? b[i][tx] : b[tx][i]) = Tb[x2 * ld + y2];
  }
  __syncthreads();
  cplx *Pb = P + o1 * sP1 + o0 * sP0;
#pragma unroll
  for (int i = ty; i < 32; i += 8) {
    const int64_t p = p0 + i, q = q0 + tx;
    if (p >= q || q >= n) continue;
    cplx v = a[i][tx];
    if (s != 0.0) { const cplx w = b[tx][i]; v.x -= s * w.x; v.y -= s * w.y; }
    cplx *dst = Pb + pair_index(p, q, n);
    *dst = axpby(ka, alpha, v, kb, beta, dst);
  }
}

__global__ void k_pair_pack(const cplx *__restrict__ T, int64_t sTo1, int64_t sTo0, int64_t sTp,
                            int64_t sTq, int64_t sTin, double s, int64_t no1, int64_t no0,
                            int64_t n, int64_t inner, cplx *P, int64_t sP1, int64_t sP0,
                            cplx alpha, int ka, cplx beta, int kb, int64_t total) {
  // iterate over (o, p, q, in) with p < q encoded through the full square; half idle
  for (int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; idx < total;
       idx += (int64_t)gridDim.x * blockDim.x) {
    int64_t in = idx % inner;
    int64_t r = idx / inner;
    int64_t q = r % n; r /= n;
    int64_t p = r % n; r /= n;
    if (p >= q) continue;
    int64_t o0 = r % no0, o1 = r / no0;
    const cplx *Tb = T + o1 * sTo1 + o0 * sTo0 + in * sTin;
    cplx v = Tb[p * sTp + q * sTq];
    if (s != 0.0) { cplx w = Tb[q * sTp + p * sTq]; v.x -= s * w.x; v.y -= s * w.y; }
    cplx *dst = P + o1 * sP1 + o0 * sP0 + pair_index(p, q, n) * inner + in;
    *dst = axpby(ka, alpha, v, kb, beta, dst);
  }
}
}  // namespace

void pair_unpack(Exec &ex, const cplx *P, int64_t no1, int64_t no0, int64_t sP1, int64_t sP0,
                 int64_t n, int64_t inner, cplx *T) {
  int64_t total = no1 * no0 * n * n * inner;
  if (total == 0) return;
  k_pair_unpack<<<grid1d(total, 256), 256, 0, ex.stream>>>(P, no1, no0, sP1, sP0, n, inner, T, total);
  ADC_CHECK_LAUNCH();
}

void pair_pack(Exec &ex, const cplx *T, int64_t sTo1, int64_t sTo0, int64_t sTp, int64_t sTq,
               int64_t sTin, double s, int64_t no1, int64_t no0, int64_t n, int64_t inner,
               cplx *P, int64_t sP1, int64_t sP0, cplx alpha, cplx beta) {
  int64_t total = no1 * no0 * n * n * inner;
  if (total == 0 || n < 2) return;
  const int ka = factor_kind(alpha), kb = factor_kind(beta);
  if (inner == 1 && (sTq == 1 || sTp == 1) && no1 * no0 <= 65535) {
    const int64_t nt = (n + 31) / 32;
    const int qfast = sTq == 1 ? 1 : 0;
    k_pair_pack_tile<<<dim3((unsigned)(nt * (nt + 1) / 2), (unsigned)(no1 * no0)), 256, 0, ex.stream>>>(
        T, sTo1, sTo0, qfast ? sTp : sTq, qfast, s, no0, n, P, sP1, sP0, alpha, ka, beta, kb);
    ADC_CHECK_LAUNCH();
    return;
  }
  k_pair_pack<<<grid1d(total, 256), 256, 0, ex.stream>>>(T, sTo1, sTo0, sTp, sTq, sTin, s, no1,
                                                         no0, n, inner, P, sP1, sP0, alpha, ka, beta, kb, total);
  ADC_CHECK_LAUNCH();
}

// ------------------------------------------------------------------ elementwise
namespace {
__global__ void k_denom2(cplx *t, const double *eo, const double *ev, int64_t o, int64_t v,
                         int64_t total) {
  for (int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; idx < total;
       idx += (int64_t)gridDim.x * blockDim.x) {
    int64_t b = idx % v, r = idx / v;
    int64_t a = r % v; r /= v;
    int64_t j = r % o, i = r / o;
    double D = eo[i] + eo[j] - ev[a] - ev[b];
    cplx x = t[idx];
    t[idx] = cmake(x.x / D, x.y / D);
  }
}
__global__ void k_denom1(cplx *t, const double *eo, const double *ev, int64_t o, int64_t v) {
  int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (idx >= o * v) return;
  int64_t a = idx % v, i = idx / v;
  double D = eo[i] - ev[a];
  cplx x = t[idx];
  t[idx] = cmake(x.x / D, x.y / D);
}
__global__ void k_oovv_from_t1(const cplx *t, const double *eo, const double *ev, int64_t o,
                               int64_t v, cplx *dst, int64_t total) {
  for (int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; idx < total;
       idx += (int64_t)gridDim.x * blockDim.x) {
    int64_t b = idx % v, r = idx / v;
    int64_t a = r % v; r /= v;
    int64_t j = r % o, i = r / o;
    double D = eo[i] + eo[j] - ev[a] - ev[b];
    cplx x = t[idx];
    dst[idx] = cmake(D * x.x, -D * x.y);
  }
}
__global__ void k_eps_diff_T(cplx *M, const cplx *G, const double *e, int64_t n, double s) {
  int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (idx >= n * n) return;
  int64_t q = idx % n, p = idx / n;
  double f = s * (e[p] - e[q]);
  cplx g = G[q * n + p];
  M[idx].x += f * g.x;
  M[idx].y += f * g.y;
}
__global__ void k_add_diag(cplx *M, const double *e, int64_t n, double s) {
  int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (p < n) M[p * n + p].x += s * e[p];
}
// g[p][q] = Re sum_Q (B_pp B_qq - B_pq B_qp): 32 columns q per block, the Cholesky index
// over eight rows of threads, summed in a fixed order
__global__ void __launch_bounds__(256)
k_antisym_diag(const cplx *B, int64_t Q, int64_t nmo, double *g) {
  __shared__ double red[8][33];
  const int64_t p = blockIdx.y, q = (int64_t)blockIdx.x * 32 + threadIdx.x;
  double acc = 0.0;
  if (q < nmo)
    for (int64_t Qi = threadIdx.y; Qi < Q; Qi += 8) {
      const cplx *Bq = B + Qi * nmo * nmo;
      const cplx pp = Bq[p * nmo + p], qq = Bq[q * nmo + q], pq = Bq[p * nmo + q], qp = Bq[q * nmo + p];
      acc += (pp.x * qq.x - pp.y * qq.y) - (pq.x * qp.x - pq.y * qp.y);
    }
  red[threadIdx.y][threadIdx.x] = acc;
  __syncthreads();
  if (threadIdx.y || q >= nmo) return;
  for (int r = 1; r < 8; ++r) acc += red[r][threadIdx.x];
  g[p * nmo + q] = acc;
}
__global__ void k_zaxpby(int64_t n, cplx a, const cplx *x, cplx b, cplx *y) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x)
    y[i] = cadd(cmul(a, x[i]), cmul(b, y[i]));
}
__global__ void k_diag_mul_add(int64_t k, int64_t n, const double *d, const cplx *x, int64_t ldx,
                               cplx *y, int64_t ldy, double s) {
  int64_t total = k * n;
  for (int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; idx < total;
       idx += (int64_t)gridDim.x * blockDim.x) {
    int64_t i = idx % n, r = idx / n;
    double f = s * d[i];
    cplx xv = x[r * ldx + i];
    cplx &yv = y[r * ldy + i];
    yv.x += f * xv.x;
    yv.y += f * xv.y;
  }
}
}  // namespace

void denom2_div(Exec &ex, cplx *t, const double *eo, const double *ev, int64_t o, int64_t v) {
  int64_t total = o * o * v * v;
  if (!total) return;
  k_denom2<<<grid1d(total, 256), 256, 0, ex.stream>>>(t, eo, ev, o, v, total);
  ADC_CHECK_LAUNCH();
}
void denom1_div(Exec &ex, cplx *t, const double *eo, const double *ev, int64_t o, int64_t v) {
  if (!o || !v) return;
  k_denom1<<<grid1d(o * v, 256), 256, 0, ex.stream>>>(t, eo, ev, o, v);
  ADC_CHECK_LAUNCH();
}
void oovv_from_t1(Exec &ex, const cplx *t, const double *eo, const double *ev, int64_t o,
                  int64_t v, cplx *dst) {
  int64_t total = o * o * v * v;
  if (!total) return;
  k_oovv_from_t1<<<grid1d(total, 256), 256, 0, ex.stream>>>(t, eo, ev, o, v, dst, total);
  ADC_CHECK_LAUNCH();
}
void add_eps_diff_transpose(Exec &ex, cplx *M, const cplx *G, const double *e, int64_t n, double s) {
  if (!n) return;
  k_eps_diff_T<<<grid1d(n * n, 256), 256, 0, ex.stream>>>(M, G, e, n, s);
  ADC_CHECK_LAUNCH();
}
void add_diag(Exec &ex, cplx *M, const double *e, int64_t n, double s) {
  if (!n) return;
  k_add_diag<<<grid1d(n, 256), 256, 0, ex.stream>>>(M, e, n, s);
  ADC_CHECK_LAUNCH();
}
void antisym_diag(Exec &ex, const cplx *B, int64_t Q, int64_t nmo, double *g) {
  // one grid row per spinor: memory ends far below 65535 of them (68 GB per Cholesky vector)
  k_antisym_diag<<<dim3((unsigned)((nmo + 31) / 32), (unsigned)nmo), dim3(32, 8), 0, ex.stream>>>(B, Q, nmo, g);
  ADC_CHECK_LAUNCH();
}
void zaxpby(Exec &ex, int64_t n, cplx a, const cplx *x, cplx b, cplx *y) {
  if (!n) return;
  k_zaxpby<<<grid1d(n, 256), 256, 0, ex.stream>>>(n, a, x, b, y);
  ADC_CHECK_LAUNCH();
}
void diag_mul_add(Exec &ex, int64_t k, int64_t n, const double *d, const cplx *x, int64_t ldx,
                  cplx *y, int64_t ldy, double s) {
  if (!k || !n) return;
  k_diag_mul_add<<<grid1d(k * n, 256), 256, 0, ex.stream>>>(k, n, d, x, ldx, y, ldy, s);
  ADC_CHECK_LAUNCH();
}

// ------------------------------------------------------------------ einsum
namespace {
struct Group {
  std::vector<char> labels;
};

// can the labels (in order) of tensor t be merged into one index with a
// uniform stride? Returns the stride of the merged index (0 if empty).
bool mergeable(const TV &t, const std::string &lab, const std::vector<char> &grp, int64_t &stride,
               int64_t &extent) {
  std::vector<std::pair<int64_t, int64_t>> es;  // (ext, str) for ext > 1
  extent = 1;
  for (char c : grp) {
    size_t pos = lab.find(c);
    int64_t e = t.ext[pos];
    extent *= e;
    if (e > 1) es.push_back({e, t.str[pos]});
  }
  if (es.empty()) { stride = 0; return true; }
  for (size_t i = 0; i + 1 < es.size(); ++i)
    if (es[i].second != es[i + 1].second * es[i + 1].first) return false;
  stride = es.back().second;
  return true;
}

// dense copy of t arranged in the concatenated label order `order`
void to_dense(Exec &ex, const TV &t, const std::string &lab, const std::vector<char> &order,
              cplx *dst) {
  std::vector<int64_t> e, s;
  for (char c : order) {
    size_t pos = lab.find(c);
    e.push_back(t.ext[pos]);
    s.push_back(t.str[pos]);
  }
  permute(ex, t.p, e, s, false, dst, C1(), C0());
}
}  // namespace

void einsum(Exec &ex, cplx alpha, const TV &A, const char *la_, const TV &B, const char *lb_,
            cplx beta, const TV &C, const char *lc_) {
  std::string la(la_), lb(lb_), lc(lc_);
  ADC_REQUIRE(la.size() == A.ext.size() && lb.size() == B.ext.size() && lc.size() == C.ext.size(),
              ADC_ERR_ARG, "einsum: label/rank mismatch " + la + "," + lb + "->" + lc);
  std::map<char, int64_t> ext;
  auto reg = [&](const std::string &l, const TV &t) {
    for (size_t i = 0; i < l.size(); ++i) {
      auto it = ext.find(l[i]);
      if (it != ext.end())
        ADC_REQUIRE(it->second == t.ext[i], ADC_ERR_ARG, std::string("einsum: extent of ") + l[i]);
      else
        ext[l[i]] = t.ext[i];
    }
  };
  reg(la, A); reg(lb, B); reg(lc, C);
  std::vector<char> gb, gm, gn, gk;
  for (char c : lc) {
    bool inA = la.find(c) != std::string::npos, inB = lb.find(c) != std::string::npos;
    ADC_REQUIRE(inA || inB, ADC_ERR_ARG, "einsum: output label not in inputs");
    if (inA && inB) gb.push_back(c);
    else if (inA) gm.push_back(c);
    else gn.push_back(c);
  }
  for (char c : la) {
    bool inB = lb.find(c) != std::string::npos, inC = lc.find(c) != std::string::npos;
    if (!inC) {
      ADC_REQUIRE(inB, ADC_ERR_UNSUPPORTED, "einsum: trace index");
      gk.push_back(c);
    }
  }
  for (char c : lb)
    ADC_REQUIRE(la.find(c) != std::string::npos || lc.find(c) != std::string::npos,
                ADC_ERR_UNSUPPORTED, "einsum: trace index in B");
  int64_t nb = 1, nm = 1, nn = 1, nk = 1;
  for (char c : gb) nb *= ext[c];
  for (char c : gm) nm *= ext[c];
  for (char c : gn) nn *= ext[c];
  for (char c : gk) nk *= ext[c];
  if (nb == 0 || nm == 0 || nn == 0) return;

  // A as [b][m][k]
  int64_t sAb, sAm, sAk, e_;
  DBuf Abuf, Bbuf, Cbuf;
  const cplx *Ap = A.p;
  if (!(mergeable(A, la, gb, sAb, e_) && mergeable(A, la, gm, sAm, e_) && mergeable(A, la, gk, sAk, e_))) {
    std::vector<char> ord(gb);
    ord.insert(ord.end(), gm.begin(), gm.end());
    ord.insert(ord.end(), gk.begin(), gk.end());
    Abuf = cbuf(ex, nb * nm * nk);
    to_dense(ex, A, la, ord, Abuf.c());
    Ap = Abuf.c();
    sAb = nm * nk; sAm = nk; sAk = 1;
  }
  int64_t sBb, sBk, sBn;
  const cplx *Bp = B.p;
  if (!(mergeable(B, lb, gb, sBb, e_) && mergeable(B, lb, gk, sBk, e_) && mergeable(B, lb, gn, sBn, e_))) {
    std::vector<char> ord(gb);
    ord.insert(ord.end(), gk.begin(), gk.end());
    ord.insert(ord.end(), gn.begin(), gn.end());
    Bbuf = cbuf(ex, nb * nk * nn);
    to_dense(ex, B, lb, ord, Bbuf.c());
    Bp = Bbuf.c();
    sBb = nk * nn; sBk = nn; sBn = 1;
  }
  int64_t sCb, sCm, sCn;
  if (mergeable(C, lc, gb, sCb, e_) && mergeable(C, lc, gm, sCm, e_) && mergeable(C, lc, gn, sCn, e_)) {
    zgemm(ex, nm, nn, nk, nb, alpha, Ap, sAb, sAm, sAk, A.conj, Bp, sBb, sBk, sBn, B.conj, beta,
          C.p, sCb, sCm, sCn);
    return;
  }
  // compute into a dense [b][m][n] buffer, then scatter into C with beta
  Cbuf = cbuf(ex, nb * nm * nn);
  zgemm(ex, nm, nn, nk, nb, alpha, Ap, sAb, sAm, sAk, A.conj, Bp, sBb, sBk, sBn, B.conj, C0(),
        Cbuf.c(), nm * nn, nn, 1);
  // C[lc] = Cbuf[perm] + beta*C: iterate C in its own label order (contiguous target
  // required for the permute kernel), so build strides of Cbuf per C label.
  std::vector<char> ord(gb);
  ord.insert(ord.end(), gm.begin(), gm.end());
  ord.insert(ord.end(), gn.begin(), gn.end());
  std::vector<int64_t> bstr(ord.size());
  {
    int64_t acc = 1;
    for (int i = (int)ord.size() - 1; i >= 0; --i) { bstr[i] = acc; acc *= ext[ord[i]]; }
  }
  // C must be contiguous for the scatter; check
  TV Cd = TV::dense(C.p, C.ext);
  ADC_REQUIRE(Cd.str == C.str, ADC_ERR_UNSUPPORTED, "einsum: non-contiguous output needs a permute");
  std::vector<int64_t> e, s;
  for (char c : lc) {
    auto it = std::find(ord.begin(), ord.end(), c);
    e.push_back(ext[c]);
    s.push_back(bstr[it - ord.begin()]);
  }
  permute(ex, Cbuf.c(), e, s, false, C.p, C1(), beta);
}

}  // namespace adc
