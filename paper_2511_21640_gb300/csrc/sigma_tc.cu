// Sigma product with the dense contractions on the tensor cores: the BF16x3
// (BF16x6) split (sigma_split) or the sliced FP64-accurate product
// (sigma_sliced, tc_slice.cu). Same terms as sigma.cu (Sec. 2.1 Eqs. 10-12);
// the coupling, ladder and ring contractions run on the tensor cores, the main
// block (n1 x n1) and the zeroth-order diagonal stay FP64.
#include <algorithm>
#include <mutex>

#include "ctx.cuh"
#include "tc_gemm.cuh"
#include "tc_slice.cuh"

namespace adc {

static void build_cache(adc_ctx *c, int planes) {
  Exec &ex = c->ex;
  auto &tc = *c->tc;
  const int64_t o = c->o, v = c->v, n1 = c->n1, n2 = c->n2;
  tc.planes = planes;
  tc_pack_A(ex, tc.Cpl, c->Cpl.c(), n1, n2, n2, 1, false, planes);
  tc_pack_A(ex, tc.CplT, c->Cpl.c(), n2, n1, 1, n2, true, planes);
  if (c->order == 3 && c->x != 0.0) {
    const int64_t P = (c->kind == ADC_EA) ? npairs(v) : npairs(o);
    if (!(c->kind == ADC_EA && c->direct_ladder)) tc_pack_A(ex, tc.Glad, c->Glad.c(), P, P, P, 1, false, planes);
    tc_pack_A(ex, tc.W, c->W.c(), o * v, o * v, o * v, 1, false, planes);
  }
  tc.err = DBuf(ex, sizeof(int));
  fill_zero(ex, tc.err.p, sizeof(int));
  tc.ready = true;
}

void release_tc(adc_ctx *c) {
  c->tc.reset();
  c->sl.reset();
}

void tc_ensure(adc_ctx *c, int planes) {
  if (c->tc && c->tc->ready && c->tc->planes < planes) c->tc.reset();  // rebuild with more planes
  if (!c->tc) c->tc.reset(new TcCache());
  if (!c->tc->ready) build_cache(c, planes);
}

namespace {
// S2[r][i] += T2[r][i] + d2[i] X2[r][i] (rows r of pitch N in S and X, n2 in T2)
__global__ void k_sat_finish(int64_t k, int64_t n2, const double *__restrict__ d2, const cplx *__restrict__ X2,
                             const cplx *__restrict__ T2, int64_t N, cplx *S2) {
  for (int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; idx < k * n2;
       idx += (int64_t)gridDim.x * blockDim.x) {
    const int64_t r = idx / n2, i = idx - r * n2;
    const cplx x = X2[r * N + i], t = T2[idx];
    cplx *s = S2 + r * N + i;
    *s = cmake(s->x + t.x + d2[i] * x.x, s->y + t.y + d2[i] * x.y);
  }
}
}  // namespace

// The BF16x3 product with every tensor-core contraction (both coupling
// directions, the satellite ladder and ring) as jobs of one persistent grouped
// launch: tiles of all terms share the SMs, so no term leaves a partly idle
// last wave, and the long-K coupling into the 1p rows is split over the SMs.
// Jobs never accumulate into the same output: the ladder writes the satellite
// rows, the coupling into them goes to a scratch block added afterwards.
static void sigma_split_grouped(adc_ctx *c, const cplx *X, cplx *S, int64_t k) {
  Exec &ex = c->ex;
  auto &tc = *c->tc;
  int *err = (int *)tc.err.p;
  const int64_t o = c->o, v = c->v, n1 = c->n1, n2 = c->n2, N = c->N;
  const bool sat = (c->order == 3 && c->x != 0.0);
  const double x = sat ? c->x : 0.0;
  const bool ea = (c->kind == ADC_EA);
  TagScope tg(ex, "main");
  zgemm(ex, k, n1, n1, 1, C1(), X, 0, N, 1, false, c->M11.c(), 0, 1, n1, false, C0(), S, 0, N, 1);
  ex.tag = "grouped";
  const int64_t nring = sat ? (ea ? k * o * v * v : k * o * v * o) : 0;
  cplx *T = scratch(c, nring + k * n2);  // ring block, then the coupling into the satellites
  cplx *T2 = T + nring;
  std::vector<TcJobDesc> jobs;
  // S1 += Cpl X2 : out[c][r] = sum_K Cpl[c][K] X2[r][K]
  tc_pack_B(ex, tc.Bx2, X + n1, k, n2, N, 0, 1, 1, false, 2);
  {
    TcJobDesc d;
    d.A = &tc.Cpl; d.B = &tc.Bx2; d.M = n1; d.N = k;
    d.alpha = C1(); d.beta = C1(); d.out = S; d.s_m = 1; d.s_nh = N; d.s_nl = 0; d.n_in = 1;
    jobs.push_back(d);
  }
  // T2 = Cpl^H X1 : out[K][r] = sum_c conj(Cpl[c][K]) X1[r][c]
  tc_pack_B(ex, tc.Bx1, X, k, n1, N, 0, 1, 1, false, 2);
  {
    TcJobDesc d;
    d.A = &tc.CplT; d.B = &tc.Bx1; d.M = n2; d.N = k;
    d.alpha = C1(); d.beta = C0(); d.out = T2; d.s_m = 1; d.s_nh = n2; d.s_nl = 0; d.n_in = 1;
    jobs.push_back(d);
  }
  if (sat) {
    if (ea) {
      const int64_t pv = npairs(v);
      // ladder: out[(ab)][(r,j)] = x sum_(cd) Glad[(ab)][(cd)] X2[r][j][(cd)], the satellite rows set
      tc_pack_B(ex, tc.Bxl, X + n1, k * o, pv, N, pv, o, 1, false, 2);
      TcJobDesc d;
      d.A = &tc.Glad; d.B = &tc.Bxl; d.M = pv; d.N = k * o;
      d.alpha = CR(x); d.beta = C0(); d.out = S + n1; d.s_m = 1; d.s_nh = N; d.s_nl = pv; d.n_in = o;
      jobs.push_back(d);
      // ring: T[r][j][a][b] = sum_(kc) W[(j,a)][(kc)] Xf[r][k][c][b]
      tc_pack_B_ring(ex, tc.Bxr, c, X, k, 2);
      TcJobDesc e;
      e.A = &tc.W; e.B = &tc.Bxr; e.M = o * v; e.N = k * v;
      e.alpha = C1(); e.beta = C0(); e.out = T; e.s_m = v; e.s_nh = o * v * v; e.s_nl = 1; e.n_in = v;
      jobs.push_back(e);
    } else {
      const int64_t po = npairs(o);
      // ladder: out[(ij)][(r,a)] = x sum_(kl) Glad[(ij)][(kl)] X2[r][(kl)][a], the satellite rows set
      tc_pack_B(ex, tc.Bxl, X + n1, k * v, po, N, 1, v, v, false, 2);
      TcJobDesc d;
      d.A = &tc.Glad; d.B = &tc.Bxl; d.M = po; d.N = k * v;
      d.alpha = CR(x); d.beta = C0(); d.out = S + n1; d.s_m = v; d.s_nh = N; d.s_nl = 1; d.n_in = v;
      jobs.push_back(d);
      // ring: T[r][j][a][i] = -sum_(kb) W[(j,a)][(kb)] Xf[r][i][k][b]
      tc_pack_B_ring(ex, tc.Bxr, c, X, k, 2);
      TcJobDesc e;
      e.A = &tc.W; e.B = &tc.Bxr; e.M = o * v; e.N = k * o;
      e.alpha = CR(-1.0); e.beta = C0(); e.out = T; e.s_m = o; e.s_nh = o * v * o; e.s_nl = 1; e.n_in = o;
      jobs.push_back(e);
    }
  } else {
    ADC_CUDA(cudaMemset2DAsync(S + n1, N * sizeof(cplx), 0, n2 * sizeof(cplx), k, ex.stream));
  }
  cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
  ADC_CUDA(cudaStreamIsCapturing(ex.stream, &cs));
  tc_gemm_grouped(ex, jobs, tc.grp, err, cs == cudaStreamCaptureStatusNone);
  ex.tag = "satellites";
  k_sat_finish<<<grid1d(k * n2, 256), 256, 0, ex.stream>>>(k, n2, c->d2.d(), X + n1, T2, N, S + n1);
  ADC_CHECK_LAUNCH();
  if (sat) {
    if (ea)
      pair_pack(ex, T, o * v * v, v * v, v, 1, 0, 1.0, k, o, v, 1, S + n1, N, npairs(v), CR(-x), C1());
    else
      pair_pack(ex, T, o * v * o, 0, 1, v * o, o, 1.0, k, 1, o, v, S + n1, N, 0, CR(x), C1());
  }
  tc_sync(ex, err);
}

void sigma_split(adc_ctx *c, const cplx *X, cplx *S, int64_t k, int nseg) {
  Exec &ex = c->ex;
  const int planes = (nseg == 6) ? 3 : 2;
  tc_ensure(c, planes);
  // the three-product split of the stored operators: one grouped launch
  if (nseg == 3 && !(c->kind == ADC_EA && c->direct_ladder) && c->opts.grouped_sigma != -1) {
    sigma_split_grouped(c, X, S, k);
    return;
  }
  auto &tc = *c->tc;
  int *err = (int *)tc.err.p;
  const int64_t o = c->o, v = c->v, n1 = c->n1, n2 = c->n2, N = c->N;
  const bool sat = (c->order == 3 && c->x != 0.0);
  const double x = sat ? c->x : 0.0;
  // S1 = X1 M11^T (FP64, n1 x n1)
  TagScope tg(ex, "main");
  zgemm(ex, k, n1, n1, 1, C1(), X, 0, N, 1, false, c->M11.c(), 0, 1, n1, false, C0(), S, 0, N, 1);
  // S1 += Cpl X2  : out[c][r] = sum_K Cpl[c][K] X2[r][K]
  ex.tag = "coupling";
  tc_pack_B(ex, tc.Bx, X + n1, k, n2, N, 0, 1, 1, false, planes);
  tc_gemm(ex, tc.Cpl, tc.Bx, n1, k, C1(), C1(), S, 1, N, 0, 1, err, nseg);
  // S2 = Cpl^H X1 : out[K][r] = sum_c conj(Cpl[c][K]) X1[r][c]
  tc_pack_B(ex, tc.Bx, X, k, n1, N, 0, 1, 1, false, planes);
  tc_gemm(ex, tc.CplT, tc.Bx, n2, k, C1(), C0(), S + n1, 1, N, 0, 1, err, nseg);
  diag_mul_add(ex, k, n2, c->d2.d(), X + n1, N, S + n1, N, 1.0);
  if (sat) {
    if (c->kind == ADC_EA) {
      const int64_t pv = npairs(v);
      // ladder: out[(ab)][(r,j)] = sum_(cd) Glad[(ab)][(cd)] X2[r][j][(cd)]
      ex.tag = "ladder";
      if (c->direct_ladder) {
        ladder_direct(c, X + n1, N, o, S + n1, N, k, x, nseg, err);
      } else {
        tc_pack_B(ex, tc.Bx, X + n1, k * o, pv, N, pv, o, 1, false, planes);
        tc_gemm(ex, tc.Glad, tc.Bx, pv, k * o, CR(x), C1(), S + n1, 1, N, pv, o, err, nseg);
      }
      // ring: T[r][j][a][b] = sum_(kc) W[(j,a)][(kc)] Xf[r][k][c][b]
      ex.tag = "ring";
      cplx *T = scratch(c, k * o * v * v);
      tc_pack_B_ring(ex, tc.Bx, c, X, k, planes);
      tc_gemm(ex, tc.W, tc.Bx, o * v, k * v, C1(), C0(), T, v, o * v * v, 1, v, err, nseg);
      pair_pack(ex, T, o * v * v, v * v, v, 1, 0, 1.0, k, o, v, 1, S + n1, N, pv, CR(-x), C1());
    } else {
      const int64_t po = npairs(o);
      // ladder: out[(ij)][(r,a)] = sum_(kl) Glad[(ij)][(kl)] X2[r][(kl)][a]
      ex.tag = "ladder";
      tc_pack_B(ex, tc.Bx, X + n1, k * v, po, N, 1, v, v, false, planes);
      tc_gemm(ex, tc.Glad, tc.Bx, po, k * v, CR(x), C1(), S + n1, v, N, 1, v, err, nseg);
      // ring: T[r][j][a][i] = -sum_(kb) W[(j,a)][(kb)] Xf[r][i][k][b]
      ex.tag = "ring";
      cplx *T = scratch(c, k * o * v * o);
      tc_pack_B_ring(ex, tc.Bx, c, X, k, planes);
      tc_gemm(ex, tc.W, tc.Bx, o * v, k * o, CR(-1.0), C0(), T, o, o * v * o, 1, o, err, nseg);
      pair_pack(ex, T, o * v * o, 0, 1, v * o, o, 1.0, k, 1, o, v, S + n1, N, 0, CR(x), C1());
    }
  }
  tc_sync(ex, err);
}

// ---- products from digits: the same contractions as sliced tensor-core products.
// Digits kept for FP64 products: all contexts of a device together at most an eighth of
// its memory (an EA problem at o = 40, v = 200 keeps 25 GB), and a context's operators
// together at most a quarter of what it has left without them.
// Any context of the device that runs short of memory takes the digits back (below).
// The lock guards the list, the totals, and whether a cache is in use: a cache that is
// not (busy 0) may lose its digits to another thread.
static std::mutex kept_mu;
static double kept_total[64];
static std::vector<SlCache *> kept_caches;

static bool kept_reserve(int dev, double bytes, double most) {
  std::lock_guard<std::mutex> lk(kept_mu);
  if (kept_total[dev] + bytes > most) return false;
  kept_total[dev] += bytes;
  return true;
}
static void kept_release(int dev, double bytes) {
  std::lock_guard<std::mutex> lk(kept_mu);
  kept_total[dev] -= bytes;
}

SlCache::SlCache(Exec &e, int d) : ex(e), dev(d) {
  std::lock_guard<std::mutex> lk(kept_mu);
  kept_caches.push_back(this);
}
SlCache::~SlCache() {
  std::lock_guard<std::mutex> lk(kept_mu);
  kept_total[dev] -= kept;
  kept_caches.erase(std::find(kept_caches.begin(), kept_caches.end(), this));
}

static int kept_dev(int dev) { return std::max(0, dev) % 64; }

void kept_digit_bytes(const adc_ctx *c, int64_t *own, int64_t *device) {
  std::lock_guard<std::mutex> lk(kept_mu);
  *own = c->sl ? (int64_t)c->sl->kept : 0;
  *device = (int64_t)kept_total[kept_dev(c->dev)];
}

size_t kept_by_others(int dev, const Exec *mine) {
  std::lock_guard<std::mutex> lk(kept_mu);
  double b = 0.0;
  for (const SlCache *sl : kept_caches)
    if (sl->dev == kept_dev(dev) && &sl->ex != mine) b += sl->kept;
  return (size_t)b;
}

// An operator whose digits found no room, or went back, is looked at again after this many
// of its products (each look asks the driver for the free memory)
constexpr int kKeepRest = 16;

// The digits kept for FP64 products alone go back (freed in the order of their context's
// stream). The lock is held; false: none kept, or the cache is in use
static bool kept_drop(SlCache &sl) {
  if (sl.busy) return false;
  bool any = false;
  for (int w = 0; w < SL_NOPS; ++w) {
    if (sl.op[w].ns * sl.op[w].b < kDigitFp64Bits) continue;
    sl.op[w] = SlMat();
    sl.rest[w] = kKeepRest;
    any = true;
  }
  kept_total[sl.dev] -= sl.kept;
  sl.kept = 0.0;
  sl.Bx = SlMat();
  sl.w.part.reset();
  return any;
}

// A context over its own limit gives its own digits back; one that finds no device memory
// takes those of every context that is not in a product: what fits without them still fits.
static bool sl_give_back(void *ctx) {
  SlCache *sl = ((adc_ctx *)ctx)->sl.get();
  if (!sl) return false;
  std::lock_guard<std::mutex> lk(kept_mu);
  return kept_drop(*sl);
}

bool reclaim_kept_digits(int dev) {
  std::lock_guard<std::mutex> lk(kept_mu);
  bool any = false;
  for (SlCache *sl : kept_caches) {
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    if (sl->dev != kept_dev(dev) || sl->busy || sl->kept <= 0.0 ||
        cudaStreamIsCapturing(sl->ex.stream, &cs) != cudaSuccess || cs != cudaStreamCaptureStatusNone)
      continue;
    // the memory is there for another stream once this one has freed it
    if (kept_drop(*sl)) any = cudaStreamSynchronize(sl->ex.stream) == cudaSuccess || any;
  }
  cudaGetLastError();
  return any;
}

static SlCache &sl_cache(adc_ctx *c) {
  if (!c->sl) {
    c->sl.reset(new SlCache(c->ex, kept_dev(c->dev)));
    c->ex.give_back = sl_give_back;
    c->ex.give_back_of = c;
  }
  return *c->sl;
}

// while it lives the cache's digits and buffers stay
struct SlUse {
  SlCache &sl;
  explicit SlUse(SlCache &s) : sl(s) {
    std::lock_guard<std::mutex> lk(kept_mu);
    ++sl.busy;
  }
  ~SlUse() {
    std::lock_guard<std::mutex> lk(kept_mu);
    --sl.busy;
  }
};

// The digits of a static operator, built when first asked for and rebuilt with
// more digits when asked for more; a product with fewer bits uses the leading
// digits of the trial vectors and the same leading digits of the operator. The shorter
// digits are cut from the longer ones' integers, so that a sliced product is the
// same whether or not an FP64 product has built these before it.
static const SlMat &sl_op(adc_ctx *c, int which, int bits) {
  Exec &ex = c->ex;
  SlMat &m = sl_cache(c).op[which];
  if (m.ns * m.b >= bits) return m;
  const int64_t o = c->o, v = c->v, n1 = c->n1, n2 = c->n2, P = (c->kind == ADC_EA) ? npairs(v) : npairs(o);
  m.ns = 0;  // nothing usable until the packing is enqueued
  SlMat t;
  std::swap(t.planes, m.planes);
  std::swap(t.exps, m.exps);
  if (which == SL_CPL) sl_pack_A(ex, t, c->Cpl.c(), n1, n2, n2, 1, false, bits, kDigitFp64Bits);
  else if (which == SL_CPLT) sl_pack_A(ex, t, c->Cpl.c(), n2, n1, 1, n2, true, bits, kDigitFp64Bits);
  else if (which == SL_GLAD) sl_pack_A(ex, t, c->Glad.c(), P, P, P, 1, false, bits, kDigitFp64Bits);
  else sl_pack_A(ex, t, c->W.c(), o * v, o * v, o * v, 1, false, bits, kDigitFp64Bits);
  m = std::move(t);
  return m;
}

void sigma_sliced(adc_ctx *c, const cplx *X, cplx *S, int64_t k, int bits) {
  ADC_REQUIRE(c->kind != ADC_EE, ADC_ERR_ARG, "sigma_sliced: IP and EA (EE goes through sigma_ee_split)");
  Exec &ex = c->ex;
  SlCache &sl = sl_cache(c);
  if (!sl.err.p) {
    sl.err = DBuf(ex, sizeof(int));
    fill_zero(ex, sl.err.p, sizeof(int));
  }
  int *err = (int *)sl.err.p;
  // One term: out = alpha op B^T + beta out, B packed by pack(op). Short of memory it gives back
  // the digits that FP64 products keep (this product needs three quarters of them) and starts
  // over: every allocation precedes the launch that writes out
  auto term = [&](int which, int64_t M, int64_t Nc, auto &&pack, cplx alpha, cplx beta, cplx *out, int64_t s_m,
                  int64_t s_nh, int64_t s_nl, int64_t n_in) {
    for (bool again = false;; again = true) {
      try {
        const SlUse use(sl);
        const SlMat &A = sl_op(c, which, kSlicedBits);
        pack(A);
        sl_gemm(ex, A, sl.Bx, M, Nc, alpha, beta, out, s_m, s_nh, s_nl, n_in, err, sl.w);
        return;
      } catch (const Error &e) {
        if (again || e.code != ADC_ERR_OOM || !sl_give_back(c)) throw;
      }
    }
  };
  auto strided = [&](const cplx *src, int64_t Nc, int64_t K, int64_t s_nh, int64_t s_nl, int64_t n_in, int64_t s_k) {
    return [=, &ex, &sl](const SlMat &A) { sl_pack_B(ex, sl.Bx, src, Nc, K, s_nh, s_nl, n_in, s_k, false, A, bits); };
  };
  auto ring = [&](const SlMat &A) { sl_pack_B_ring(ex, sl.Bx, c, X, k, A, bits); };
  const int64_t o = c->o, v = c->v, n1 = c->n1, n2 = c->n2, N = c->N;
  const bool sat = (c->order == 3 && c->x != 0.0);
  const double x = sat ? c->x : 0.0;
  // S1 = X1 M11^T (FP64, n1 x n1)
  TagScope tg(ex, "main");
  zgemm(ex, k, n1, n1, 1, C1(), X, 0, N, 1, false, c->M11.c(), 0, 1, n1, false, C0(), S, 0, N, 1);
  // S1 += Cpl X2, S2 = Cpl^H X1
  ex.tag = "coupling";
  term(SL_CPL, n1, k, strided(X + n1, k, n2, N, 0, 1, 1), C1(), C1(), S, 1, N, 0, 1);
  term(SL_CPLT, n2, k, strided(X, k, n1, N, 0, 1, 1), C1(), C0(), S + n1, 1, N, 0, 1);
  diag_mul_add(ex, k, n2, c->d2.d(), X + n1, N, S + n1, N, 1.0);
  if (sat) {
    if (c->kind == ADC_EA) {
      const int64_t pv = npairs(v);
      ex.tag = "ladder";
      if (c->direct_ladder) {
        ladder_direct(c, X + n1, N, o, S + n1, N, k, x, ADC_LADDER_SLICED, err);
      } else {
        term(SL_GLAD, pv, k * o, strided(X + n1, k * o, pv, N, pv, o, 1), CR(x), C1(), S + n1, 1, N, pv, o);
      }
      ex.tag = "ring";
      cplx *T = scratch(c, k * o * v * v);
      term(SL_W, o * v, k * v, ring, C1(), C0(), T, v, o * v * v, 1, v);
      pair_pack(ex, T, o * v * v, v * v, v, 1, 0, 1.0, k, o, v, 1, S + n1, N, pv, CR(-x), C1());
    } else {
      const int64_t po = npairs(o);
      ex.tag = "ladder";
      term(SL_GLAD, po, k * v, strided(X + n1, k * v, po, N, 1, v, v), CR(x), C1(), S + n1, v, N, 1, v);
      ex.tag = "ring";
      cplx *T = scratch(c, k * o * v * o);
      term(SL_W, o * v, k * o, ring, CR(-1.0), C0(), T, o, o * v * o, 1, o);
      pair_pack(ex, T, o * v * o, 0, 1, v * o, o, 1.0, k, 1, o, v, S + n1, N, 0, CR(x), C1());
    }
  }
  tc_sync(ex, err);
}

// the kept FP64 digits of an operator (M x K), built when there is room for them; null: none kept
static const SlMat *sl_kept_op(adc_ctx *c, SlCache &sl, int which, int64_t M, int64_t K) {
  SlMat &m = sl.op[which];
  if (m.ns * m.b >= kDigitFp64Bits) return &m;
  if (!c->keep_digits) return nullptr;
  if (sl.rest[which] > 0) {
    --sl.rest[which];
    return nullptr;
  }
  const double need = 4.0 * sl_digits(K, kDigitFp64Bits).ns * (double)M * (double)sl_kp(K);
  double room = (double)unused_device_memory();
  if (c->ex.mem_limit > 0) room = std::min(room, (double)(c->ex.mem_limit - c->ex.mem_used));
  size_t fr = 0, tot = 0;
  ADC_CUDA(cudaMemGetInfo(&fr, &tot));
  sl.rest[which] = kKeepRest;
  const OptionalAlloc opt(c->ex);
  if (sl.kept + need > 0.25 * (room + sl.kept) || !kept_reserve(sl.dev, need, 0.125 * (double)tot)) return nullptr;
  try {
    sl_op(c, which, kDigitFp64Bits);
  } catch (const Error &e) {
    kept_release(sl.dev, need);
    if (e.code != ADC_ERR_OOM) throw;
    return nullptr;
  }
  {
    std::lock_guard<std::mutex> lk(kept_mu);
    sl.kept += need;
  }
  sl.rest[which] = 0;
  return &m;
}

// ---- one term of the FP64 product with the kept digits of its operator:
// out = alpha op B^T + beta out as tc_gemm addresses it, B by its strides or (ring)
// gathered from X2. Slicing the operator again in every product took 6.9 of the
// 23.6 ms of device time of an EA product at o = 30, v = 150, 8 vectors, and 4.0 of
// 7.0 ms at second order (o = 25, v = 180, 6 vectors). False (nothing enqueued to out):
// the term is small, the stream is capturing, or the digits do not fit.
bool fp64_op_product(adc_ctx *c, int which, bool ring, const cplx *X, int64_t k, const cplx *Bsrc, int64_t Nc,
                     int64_t b_nh, int64_t b_nl, int64_t b_in, int64_t b_k, cplx alpha, cplx beta, cplx *out,
                     int64_t s_m, int64_t s_nh, int64_t s_nl, int64_t n_in) {
  Exec &ex = c->ex;
  const int64_t o = c->o, v = c->v, n1 = c->n1, n2 = c->n2, P = (c->kind == ADC_EA) ? npairs(v) : npairs(o);
  const int64_t M = which == SL_CPL ? n1 : which == SL_CPLT ? n2 : which == SL_GLAD ? P : o * v;
  const int64_t K = which == SL_CPL ? n2 : which == SL_CPLT ? n1 : M;
  if (!fp64_digits_usable(ex, M, Nc, K)) return false;
  SlCache &sl = sl_cache(c);
  const SlUse use(sl);
  // (the whole block is sliced at once)
  const double bx = 8.0 * sl_digits(K, kDigitFp64Bits).ns * (double)Nc * (double)sl_kp(K);
  if (ex.digit_limit > 0 && bx > 0.375 * (double)ex.digit_limit) return false;
  const SlMat *op = sl_kept_op(c, sl, which, M, K);
  if (!op) return false;
  const OptionalAlloc opt(ex);
  try {
    const SlMat &A = *op;
    if (ring) sl_pack_B_ring(ex, sl.Bx, c, X, k, A, kDigitFp64Bits);
    else sl_pack_B(ex, sl.Bx, Bsrc, Nc, K, b_nh, b_nl, b_in, b_k, false, A, kDigitFp64Bits);
    sl_gemm(ex, A, sl.Bx, M, Nc, alpha, beta, out, s_m, s_nh, s_nl, n_in, ex.digit_err, sl.w);
  } catch (const Error &e) {
    if (e.code != ADC_ERR_OOM) throw;
    return false;
  }
  return true;
}

// the operators' digits that an FP64 product of k vectors will use, built ahead
// of a solve that takes the memory left (a term too small to use them builds none)
void fp64_ops_prepare(adc_ctx *c, int64_t k) {
  if (c->kind == ADC_EE) return;
  const int64_t o = c->o, v = c->v, n1 = c->n1, n2 = c->n2, P = (c->kind == ADC_EA) ? npairs(v) : npairs(o);
  const bool ea = (c->kind == ADC_EA), sat = (c->order == 3 && c->x != 0.0);
  const int64_t M[SL_NOPS] = {n1, n2, P, o * v}, K[SL_NOPS] = {n2, n1, P, o * v};
  const int64_t Nc[SL_NOPS] = {k, k, k * (ea ? o : v), k * (ea ? v : o)};
  for (int w = 0; w < SL_NOPS; ++w) {
    if (w >= SL_GLAD && !sat) continue;
    if (w == SL_GLAD && ea && c->direct_ladder) continue;
    if (!fp64_digits_usable(c->ex, M[w], Nc[w], K[w])) continue;
    SlCache &sl = sl_cache(c);
    const SlUse use(sl);
    sl_kept_op(c, sl, w, M[w], K[w]);
  }
}

}  // namespace adc
