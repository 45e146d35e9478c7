// Small dense Hermitian eigensolver on the device: cyclic Jacobi with the
// round-robin ordering (disjoint pairs rotated in parallel), FP64, one CTA.
// Used for the Rayleigh-Ritz step of Davidson (Eq. 10 projected onto the
// subspace) and for the natural-spinor and semicanonical diagonalisations
// (Eqs. 26 and 29).
#include "eig.cuh"

namespace adc {

namespace {

__device__ inline double block_sum(double v, double *red) {
  for (int off = 16; off > 0; off >>= 1) v += __shfl_down_sync(0xffffffffu, v, off);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  __syncthreads();
  if (lane == 0) red[wid] = v;
  __syncthreads();
  if (wid == 0) {
    v = (lane < (int)(blockDim.x >> 5)) ? red[lane] : 0.0;
    for (int off = 16; off > 0; off >>= 1) v += __shfl_down_sync(0xffffffffu, v, off);
    if (lane == 0) red[0] = v;
  }
  __syncthreads();
  double r = red[0];
  __syncthreads();
  return r;
}

// A (n x n, leading dimension lda) is overwritten; eigenvalues ascending into
// w, eigenvectors as columns of Vout (leading dimension ldv). Vwork n x n.
// info[0] = sweeps used, or -1 when the sweep limit was reached.
// With in_smem the matrix and the eigenvector work array live in shared
// memory for the whole iteration (n up to about 80), else in global memory.
__global__ void __launch_bounds__(1024)
k_jacobi(cplx *Ag, int n, int ldag, cplx *Vg, double *w, cplx *Vout, int ldv, int *info,
         int max_sweeps, double rel_tol, int in_smem) {
  extern __shared__ double sm[];
  const int np = n + (n & 1);       // even number of players
  const int npairs = np / 2;
  double *rc = sm;                  // cos per pair
  double *rs = rc + npairs;         // sin per pair
  double *rpr = rs + npairs;        // phase re
  double *rpi = rpr + npairs;       // phase im
  int *pp = (int *)(rpi + npairs);
  int *pq = pp + npairs;
  double *red = (double *)(pq + npairs);
  const int tid = threadIdx.x, nt = blockDim.x;
  cplx *A = Ag, *Vwork = Vg;
  int lda = ldag;
  if (in_smem) {
    // after the 64 reduction slots, 16-byte aligned
    uintptr_t base = ((uintptr_t)(red + 64) + 15) & ~(uintptr_t)15;
    A = (cplx *)base;
    Vwork = A + (int64_t)n * n;
    lda = n;
    for (int idx = tid; idx < n * n; idx += nt) A[idx] = Ag[(int64_t)(idx / n) * ldag + idx % n];
    __syncthreads();
  }

  for (int idx = tid; idx < n * n; idx += nt) {
    int r = idx / n, cI = idx % n;
    Vwork[(int64_t)r * n + cI] = cmake(r == cI ? 1.0 : 0.0, 0.0);
  }
  // Frobenius norm for the stopping test
  double loc = 0.0;
  for (int idx = tid; idx < n * n; idx += nt) {
    cplx a = A[(int64_t)(idx / n) * lda + idx % n];
    loc += a.x * a.x + a.y * a.y;
  }
  const double fro2 = block_sum(loc, red);
  int sweeps = 0;
  bool done = (n <= 1);
  while (!done && sweeps < max_sweeps) {
    for (int step = 0; step < np - 1; ++step) {
      // pairs of this round
      for (int k = tid; k < npairs; k += nt) {
        int a = (k == 0) ? 0 : ((k - 1 + step) % (np - 1)) + 1;
        int kb = np - 1 - k;
        int b = ((kb - 1 + step) % (np - 1)) + 1;
        int p = min(a, b), q = max(a, b);
        pp[k] = p;
        pq[k] = q;
        double cs = 1.0, sn = 0.0, er = 1.0, ei = 0.0;
        if (q < n) {
          double app = A[(int64_t)p * lda + p].x, aqq = A[(int64_t)q * lda + q].x;
          cplx apq = A[(int64_t)p * lda + q];
          double mag = sqrt(apq.x * apq.x + apq.y * apq.y);
          if (mag > 1e-300) {
            er = apq.x / mag;
            ei = apq.y / mag;
            double tau = (aqq - app) / (2.0 * mag);
            double t = (tau >= 0.0 ? 1.0 : -1.0) / (fabs(tau) + sqrt(1.0 + tau * tau));
            cs = 1.0 / sqrt(1.0 + t * t);
            sn = t * cs;
          }
        }
        rc[k] = cs; rs[k] = sn; rpr[k] = er; rpi[k] = ei;
      }
      __syncthreads();
      // rows: new row p = cs A[p,:] - sn e^{i phi} A[q,:]; row q = sn A[p,:] + cs e^{i phi} A[q,:]
      for (int idx = tid; idx < npairs * n; idx += nt) {
        int k = idx / n, col = idx % n;
        int p = pp[k], q = pq[k];
        if (q >= n) continue;
        double cs = rc[k], sn = rs[k];
        cplx e = cmake(rpr[k], rpi[k]);
        cplx ap = A[(int64_t)p * lda + col], aq = A[(int64_t)q * lda + col];
        cplx eaq = cmul(e, aq);
        A[(int64_t)p * lda + col] = cmake(cs * ap.x - sn * eaq.x, cs * ap.y - sn * eaq.y);
        A[(int64_t)q * lda + col] = cmake(sn * ap.x + cs * eaq.x, sn * ap.y + cs * eaq.y);
      }
      __syncthreads();
      // columns (A and V): new col p = cs X[:,p] - sn e^{-i phi} X[:,q]; col q = sn X[:,p] + cs e^{-i phi} X[:,q]
      for (int idx = tid; idx < npairs * n * 2; idx += nt) {
        int which = idx / (npairs * n);
        int rem = idx % (npairs * n);
        int k = rem / n, row = rem % n;
        int p = pp[k], q = pq[k];
        if (q >= n) continue;
        double cs = rc[k], sn = rs[k];
        cplx ec = cmake(rpr[k], -rpi[k]);
        cplx *X = which ? Vwork : A;
        int64_t ld = which ? n : lda;
        cplx xp = X[(int64_t)row * ld + p], xq = X[(int64_t)row * ld + q];
        cplx exq = cmul(ec, xq);
        X[(int64_t)row * ld + p] = cmake(cs * xp.x - sn * exq.x, cs * xp.y - sn * exq.y);
        X[(int64_t)row * ld + q] = cmake(sn * xp.x + cs * exq.x, sn * xp.y + cs * exq.y);
      }
      __syncthreads();
    }
    ++sweeps;
    double off = 0.0;
    for (int idx = tid; idx < n * n; idx += nt) {
      int r = idx / n, cI = idx % n;
      if (r != cI) {
        cplx a = A[(int64_t)r * lda + cI];
        off += a.x * a.x + a.y * a.y;
      }
    }
    off = block_sum(off, red);
    done = (off <= rel_tol * rel_tol * fro2) || (off == 0.0);
  }
  // sort ascending by rank counting (ties broken by index)
  for (int i = tid; i < n; i += nt) {
    double di = A[(int64_t)i * lda + i].x;
    int rank = 0;
    for (int j = 0; j < n; ++j) {
      double dj = A[(int64_t)j * lda + j].x;
      if (dj < di || (dj == di && j < i)) ++rank;
    }
    w[rank] = di;
    for (int r = 0; r < n; ++r) Vout[(int64_t)r * ldv + rank] = Vwork[(int64_t)r * n + i];
  }
  if (in_smem) {
    __syncthreads();
    // the diagonalised matrix back to the caller's array (its diagonal holds the eigenvalues)
    for (int idx = tid; idx < n * n; idx += nt) Ag[(int64_t)(idx / n) * ldag + idx % n] = A[idx];
  }
  if (tid == 0) info[0] = done ? sweeps : -1;
}

// ---------------------------------------------------------------- FP32 start + FP64 refinement
// For the Rayleigh-Ritz steps of the Davidson solver (n up to 128) one SM's
// FP64 units (two FMAs per clock) make an FP64 Jacobi take milliseconds.
// Instead: (1) cyclic Jacobi in FP32 on A - sigma I (sigma the mean diagonal),
// one CTA, to about 1e-7 of the spectrum's spread; (2) FP64 iterative
// refinement of the whole eigendecomposition after Ogita and Aishima (2018):
// with X the current eigenvectors, H = X^H X and S = X^H (A - sigma) X (both
// made exactly Hermitian), R = I - H,
//   lambda_i = S_ii / H_ii,
//   F_ij = (S_ij + lambda_j R_ij) / (lambda_j - lambda_i)   for separated i, j,
//          R_ij / 2                                         within a cluster and for i = j,
//   X <- X (I + F),
// which converges quadratically for separated eigenvalues. Hermitian S and H
// make F_ij + conj(F_ji) = R_ij exactly, so the update keeps X orthonormal to
// second order whatever the gap. Columns are coupled when their gap is below
// delta = 2 (||S - diag S||_F + max|lambda| ||R||_F) (the bound of the method),
// below 1e-8 max|lambda| (gaps the FP64 products resolve too coarsely), or when the
// first-order correction would exceed 1e-3 (its second-order error would not
// be small); clusters are the connected components of the coupling. Each
// cluster of at most CL_MAX columns is diagonalised exactly: the FP64 Jacobi
// eigenvectors U of P^H S_c P (P = I + R_c / 2, the first-order Loewdin
// factor of its non-orthonormal basis) rotate its columns of I + F, and their
// eigenvalues replace its lambda. The host repeats steps until the
// corrections between clusters are below 1e-8 of the gaps (beyond the
// rounding noise of S) and the updated X is orthonormal to 1e-13, at least
// nsteps and at most nsteps + 3; otherwise (a cluster wider than CL_MAX, no
// convergence) the FP64 Jacobi solves the matrix instead. The n^3 products
// run as small FP64 GEMMs over many SMs.

constexpr int EIG_NMAX = 128;
constexpr int CL_MAX = 8;
constexpr double OA_ETA = 1e-3;   // largest first-order correction between separate clusters
// gaps below this fraction of max|lambda| always couple: beyond it the rounding
// of S (about eps |lambda|) gives first-order corrections below 1e-8, whose
// squares stay below the rounding of an orthonormal basis
constexpr double OA_TAU = 1e-8;
constexpr double OA_ORTH = 1e-13;  // largest |X^H X - I| of an accepted decomposition

__device__ inline float2 f2mul(float2 a, float2 b) { return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x); }

// (x, y) <- (cs x - sn e y, sn x + cs e y)
__device__ inline void turn(float2 &x, float2 &y, float cs, float sn, float2 e) {
  const float2 ey = f2mul(e, y);
  y = make_float2(sn * x.x + cs * ey.x, sn * x.y + cs * ey.y);
  x = make_float2(cs * x.x - sn * ey.x, cs * x.y - sn * ey.y);
}

__device__ inline float block_sum_f(float v, float *red) {
  for (int off = 16; off > 0; off >>= 1) v += __shfl_down_sync(0xffffffffu, v, off);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  __syncthreads();
  if (lane == 0) red[wid] = v;
  __syncthreads();
  if (wid == 0) {
    v = (lane < (int)(blockDim.x >> 5)) ? red[lane] : 0.f;
    for (int off = 16; off > 0; off >>= 1) v += __shfl_down_sync(0xffffffffu, v, off);
    if (lane == 0) red[0] = v;
  }
  __syncthreads();
  float r = red[0];
  __syncthreads();
  return r;
}

__device__ inline double block_max(double v, double *red) {
  for (int off = 16; off > 0; off >>= 1) v = fmax(v, __shfl_down_sync(0xffffffffu, v, off));
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  __syncthreads();
  if (lane == 0) red[wid] = v;
  __syncthreads();
  if (wid == 0) {
    v = (lane < (int)(blockDim.x >> 5)) ? red[lane] : 0.0;
    for (int off = 16; off > 0; off >>= 1) v = fmax(v, __shfl_down_sync(0xffffffffu, v, off));
    if (lane == 0) red[0] = v;
  }
  __syncthreads();
  double r = red[0];
  __syncthreads();
  return r;
}

// shared memory of k_jacobi32 before the matrices (rotation tables, pair lists, reduction)
__host__ __device__ inline size_t jacobi32_head_bytes(int n) {
  const int np = n + (n & 1);
  return (size_t)np / 2 * 4 * sizeof(float) + (size_t)np * sizeof(int) + 64 * sizeof(float) + 16;
}

// A (FP64, lda) -> FP32 A - sigma I in shared memory; cyclic Jacobi (round robin);
// eigenvectors sorted by ascending eigenvalue into X (FP64, n x n, columns), sigma
// into *shift. The eigenvector work array (transposed: one row per vector) lives in
// shared memory, or in Vg (n x n FP32 complex in global memory) when Vg is given.
// What bounds it: the chain of np - 1 steps per sweep, each a barrier, the angles, a
// barrier and the rotations. Pairs are disjoint, so the 2 x 2 block of pair k's rows
// and pair l's columns needs only its own four elements: one thread turns it from
// both sides, in one pass over A and without the barrier between rows and columns.
// A warp owns a pair k of A or of the vectors, so no index is divided.
// Measured over the solves of an IP o=8 v=24 Davidson (n up to 48): 174 -> 122 us a call.
__global__ void __launch_bounds__(1024)
k_jacobi32(const cplx *__restrict__ Ag, int n, int lda, cplx *X, double *shift, int max_sweeps, float2 *Vg) {
  extern __shared__ float smf[];
  const int np = n + (n & 1), npairs = np / 2;
  float *rc = smf, *rs = rc + npairs, *rpr = rs + npairs, *rpi = rpr + npairs;
  int *pp = (int *)(rpi + npairs), *pq = pp + npairs;
  float *red = (float *)(pq + npairs);
  // rows padded to n + 1 elements: reads down a column (the last pass over V) are free
  // of bank conflicts
  const int ld = n + 1;
  float2 *A = (float2 *)(((uintptr_t)(red + 64) + 15) & ~(uintptr_t)15);
  float2 *V = Vg ? Vg : A + n * ld;
  __shared__ double dred[32];
  const int tid = threadIdx.x, nt = blockDim.x;
  const int lane = tid & 31, wid = tid >> 5, nw = nt >> 5;
  // shift by the mean diagonal (FP64), then round
  double ds = 0.0;
  for (int i = tid; i < n; i += nt) ds += Ag[(int64_t)i * lda + i].x;
  for (int off = 16; off > 0; off >>= 1) ds += __shfl_down_sync(0xffffffffu, ds, off);
  if ((tid & 31) == 0) dred[tid >> 5] = ds;
  __syncthreads();
  if (tid == 0) {
    double t = 0.0;
    for (int w = 0; w < (nt >> 5); ++w) t += dred[w];
    dred[0] = t / n;
  }
  __syncthreads();
  const double sigma = dred[0];
  for (int idx = tid; idx < n * n; idx += nt) {
    const int r = idx / n, c = idx % n;
    const cplx a = Ag[(int64_t)r * lda + c];
    A[r * ld + c] = make_float2((float)(a.x - (r == c ? sigma : 0.0)), (float)a.y);
    V[r * ld + c] = make_float2(r == c ? 1.f : 0.f, 0.f);
  }
  __syncthreads();
  float loc = 0.f;
  for (int idx = tid; idx < n * n; idx += nt) {
    const float2 a = A[(idx / n) * ld + idx % n];
    loc += a.x * a.x + a.y * a.y;
  }
  const float fro2 = block_sum_f(loc, red);
  bool done = (n <= 1);
  float prev = 3.0e38f;
  for (int sweep = 0; !done && sweep < max_sweeps; ++sweep) {
    for (int step = 0; step < np - 1; ++step) {
      for (int k = tid; k < npairs; k += nt) {
        const int m = np - 1, ka = k - 1 + step, kb = np - 2 - k + step;   // both below 2 m
        const int a = (k == 0) ? 0 : (ka < m ? ka : ka - m) + 1;
        const int b = (kb < m ? kb : kb - m) + 1;
        const int p = min(a, b), q = max(a, b);
        pp[k] = p;
        pq[k] = q;
        float cs = 1.f, sn = 0.f, er = 1.f, ei = 0.f;
        if (q < n) {
          const float app = A[p * ld + p].x, aqq = A[q * ld + q].x;
          const float2 apq = A[p * ld + q];
          const float mag = sqrtf(apq.x * apq.x + apq.y * apq.y);
          if (mag > 1e-30f) {
            er = apq.x / mag;
            ei = apq.y / mag;
            const float tau = (aqq - app) / (2.f * mag);
            const float t = (tau >= 0.f ? 1.f : -1.f) / (fabsf(tau) + sqrtf(1.f + tau * tau));
            cs = 1.f / sqrtf(1.f + t * t);
            sn = t * cs;
          }
        }
        rc[k] = cs; rs[k] = sn; rpr[k] = er; rpi[k] = ei;
      }
      __syncthreads();
      for (int task = wid; task < 2 * npairs; task += nw) {
        const int k = task < npairs ? task : task - npairs;
        const int p = pp[k], q = pq[k];
        const float cs = rc[k], sn = rs[k];
        const float2 e = make_float2(rpr[k], rpi[k]);
        if (task >= npairs) {   // vectors p and q
          if (q >= n) continue;
          for (int c = lane; c < n; c += 32) {
            float2 x = V[p * ld + c], y = V[q * ld + c];
            turn(x, y, cs, sn, make_float2(e.x, -e.y));
            V[p * ld + c] = x;
            V[q * ld + c] = y;
          }
          continue;
        }
        for (int l = lane; l < npairs; l += 32) {
          const int pl = pp[l], ql = pq[l];
          const bool hq = q < n, hl = ql < n;
          const float2 z = make_float2(0.f, 0.f);
          float2 a00 = A[p * ld + pl], a01 = hl ? A[p * ld + ql] : z;
          float2 a10 = hq ? A[q * ld + pl] : z, a11 = hq && hl ? A[q * ld + ql] : z;
          if (hq) {
            turn(a00, a10, cs, sn, e);
            turn(a01, a11, cs, sn, e);
          }
          if (hl) {
            const float2 ec = make_float2(rpr[l], -rpi[l]);
            turn(a00, a01, rc[l], rs[l], ec);
            turn(a10, a11, rc[l], rs[l], ec);
            A[p * ld + ql] = a01;
          }
          A[p * ld + pl] = a00;
          if (hq) {
            A[q * ld + pl] = a10;
            if (hl) A[q * ld + ql] = a11;
          }
        }
      }
      __syncthreads();
    }
    float off = 0.f;
    for (int idx = tid; idx < n * n; idx += nt) {
      const int r = idx / n, c = idx % n;
      if (r != c) off += A[r * ld + c].x * A[r * ld + c].x + A[r * ld + c].y * A[r * ld + c].y;
    }
    off = block_sum_f(off, red);
    // converged, or at the FP32 rounding floor (the off-diagonal norm no longer drops)
    done = (off <= 1e-13f * fro2) || (off == 0.f) || (off <= 1e-9f * fro2 && sweep >= 1 && off > 0.25f * prev);
    prev = off;
  }
  // columns sorted by ascending eigenvalue, promoted to FP64
  for (int i = tid; i < n; i += nt) {
    const float di = A[i * ld + i].x;
    int rank = 0;
    for (int j = 0; j < n; ++j) {
      const float dj = A[j * ld + j].x;
      if (dj < di || (dj == di && j < i)) ++rank;
    }
    for (int r = 0; r < n; ++r) X[(int64_t)r * n + rank] = cmake((double)V[i * ld + r].x, (double)V[i * ld + r].y);
  }
  if (tid == 0) *shift = sigma;
}

// C = op(A) B (n x n, FP64): 8 x 8 output tile per CTA, A rows and B columns of the
// tile staged in shared memory; opA: 0 = A, 1 = A^H; with shift, A - shift I is used
// for A (opA = 0). herm: C is Hermitian, tiles below the diagonal are the conjugates
// of those above. blockIdx.z picks one of two independent products. Two warps per half
// of k: at 64 clocks per FP64 warp instruction of an SM's quarter, the four quarters
// have to share a tile. With H and T in one launch and the
// mirrored tiles, a step's products took 23 -> 14 us at n up to 48.
constexpr int SG_T = 8, SG_THREADS = 2 * SG_T * SG_T;
struct SgArgs {
  const cplx *A;
  int lda, opA;
  const double *shift;
  const cplx *B;
  cplx *C;
  int herm;
};
__global__ void __launch_bounds__(SG_THREADS)
k_small_gemm(SgArgs g0, SgArgs g1, int n) {
  extern __shared__ double smg[];
  __shared__ cplx half_sum[SG_T * SG_T];
  const SgArgs g = blockIdx.z ? g1 : g0;
  if (g.herm && blockIdx.x < blockIdx.y) return;
  cplx *sa = (cplx *)smg;            // [SG_T][n] rows i of op(A)
  cplx *sb = sa + SG_T * n;          // [n][SG_T] columns j of B
  const int i0 = blockIdx.y * SG_T, j0 = blockIdx.x * SG_T;
  const double sh = g.shift ? *g.shift : 0.0;
  for (int e = threadIdx.x; e < SG_T * n; e += SG_THREADS) {
    const int kt = e / SG_T, t = e % SG_T;
    cplx a = cmake(0.0, 0.0);
    if (g.opA) {
      const int i = i0 + t;
      if (i < n) { a = g.A[(int64_t)kt * g.lda + i]; a.y = -a.y; }
      sa[t * n + kt] = a;
    } else {
      const int ii = e / n, k = e % n, i = i0 + ii;
      if (i < n) { a = g.A[(int64_t)i * g.lda + k]; if (k == i) a.x -= sh; }
      sa[e] = a;
    }
    sb[e] = (j0 + t < n) ? g.B[(int64_t)kt * n + j0 + t] : cmake(0.0, 0.0);
  }
  __syncthreads();
  const int half = threadIdx.x / (SG_T * SG_T), t = threadIdx.x % (SG_T * SG_T);
  const int ii = t / SG_T, jj = t % SG_T;
  const int i = i0 + ii, j = j0 + jj;
  double re = 0.0, im = 0.0;
  const int kh = (n + 1) / 2, k1 = half ? n : kh;
  for (int k = half ? kh : 0; k < k1; ++k) {
    const cplx a = sa[ii * n + k], b = sb[k * SG_T + jj];
    re = fma(a.x, b.x, re);
    re = fma(-a.y, b.y, re);
    im = fma(a.x, b.y, im);
    im = fma(a.y, b.x, im);
  }
  if (half) half_sum[t] = cmake(re, im);
  __syncthreads();
  if (half || i >= n || j >= n) return;
  const cplx r = cadd(cmake(re, im), half_sum[t]);
  g.C[(int64_t)i * n + j] = r;
  if (g.herm && blockIdx.x > blockIdx.y) g.C[(int64_t)j * n + i] = cconj(r);
}

// Hermitian part of M (n x n) at (i, j)
__device__ inline cplx herm_at(const cplx *__restrict__ M, int n, int i, int j) {
  const cplx a = M[(int64_t)i * n + j], b = M[(int64_t)j * n + i];
  return cmake(0.5 * (a.x + b.x), 0.5 * (a.y - b.y));
}

// One refinement step: from H = X^H X and S = X^H (A - shift) X the estimates lam, the
// clusters and F = I + correction, with every cluster's columns turned by its
// eigenvectors. Some 40 FP64 operations per element: one SM's FP64 units (two fused
// multiply-adds per clock) need longer for them than all SMs for the products, so four
// launches spread them by rows; what a step needs of the whole matrix (norms, coupling
// bits, labels) goes through a few kilobytes of scratch, and each CTA reads all of it.
// Measured in the same Davidson: 75 -> 21 us a step, of which eight-column clusters
// (one thread's Jacobi of 1.3 ms before) now at most 61 us. The whole eigensolver, random
// spectrum: n = 32 0.60 -> 0.37 ms, 64 2.20 -> 1.04, 96 5.45 -> 2.60, 128 20.3 -> 6.9.
constexpr int OA_W = EIG_NMAX / 32;
constexpr int OA_PARTS = EIG_NMAX;    // one CTA per row
struct OaArgs {
  const cplx *H, *S;
  int n;
  double *rq;               // [n] Rayleigh quotients S_ii / H_ii
  double *lam;              // [n] out: eigenvalue estimates
  double *part;             // [2][OA_PARTS] per-row sums of |S_ij|^2 (i != j) and |R_ij|^2
  unsigned *mask;           // [n][OA_W] coupling bits
  cplx *U;                  // [n][CL_MAX] row j: j's row of its cluster's eigenvectors
  int *label;               // [n] smallest column of the column's cluster
  double *stat;             // [0]: largest (|num_ij| - 1e-14 max|lam|) / |gap_ij| over pairs
                            // in different clusters; [1]: clusters wider than CL_MAX
  cplx *F;
};

// row blockIdx.x: Rayleigh quotient and norms
__global__ void __launch_bounds__(EIG_NMAX)
k_oa_norms(OaArgs o) {
  __shared__ double red[32];
  const int n = o.n, i = blockIdx.x, j = threadIdx.x;
  double so = 0.0, rr = 0.0;
  if (j < n) {
    const cplx h = herm_at(o.H, n, i, j);
    const double rx = (i == j ? 1.0 : 0.0) - h.x, ry = -h.y;
    rr = rx * rx + ry * ry;
    if (i != j) {
      const cplx sv = herm_at(o.S, n, i, j);
      so = sv.x * sv.x + sv.y * sv.y;
    }
  }
  so = block_sum(so, red);
  rr = block_sum(rr, red);
  if (j == 0) {
    o.part[i] = so;
    o.part[OA_PARTS + i] = rr;
    o.rq[i] = o.S[(int64_t)i * n + i].x / o.H[(int64_t)i * n + i].x;
    if (i == 0) o.stat[0] = 0.0;
  }
}

// row blockIdx.x of the coupling bits
__global__ void __launch_bounds__(EIG_NMAX)
k_oa_couple(OaArgs o) {
  __shared__ double red[32];
  const int n = o.n, i = blockIdx.x, j = threadIdx.x;
  const double so = block_sum(j < n ? o.part[j] : 0.0, red);
  const double rr = block_sum(j < n ? o.part[OA_PARTS + j] : 0.0, red);
  const double lm = block_max(j < n ? fabs(o.rq[j]) : 0.0, red);
  const double thr = fmax(2.0 * (sqrt(so) + lm * sqrt(rr)), OA_TAU * lm);
  bool couple = false;
  if (j < n && j != i) {
    const int a = min(i, j), b = max(i, j);
    const cplx h = herm_at(o.H, n, a, b), sv = herm_at(o.S, n, a, b);
    const double lb = o.rq[b], gap = lb - o.rq[a];
    const double nx = sv.x - lb * h.x, ny = sv.y - lb * h.y;   // S_ab + lam_b R_ab
    couple = fabs(gap) <= thr || OA_ETA * fabs(gap) <= sqrt(nx * nx + ny * ny);
  }
  const unsigned bits = __ballot_sync(0xffffffffu, couple);
  if ((j & 31) == 0) o.mask[i * OA_W + (j >> 5)] = bits;
}

// connected components of the coupling: every column takes the smallest label among
// its neighbours until nothing changes (labels only decrease). One thread per column.
__device__ inline void oa_labels(const unsigned *mask, int n, int *lab) {
  const int j = threadIdx.x;
  unsigned m[OA_W];
  for (int w = 0; w < OA_W; ++w) m[w] = j < n ? mask[j * OA_W + w] : 0u;
  lab[j] = j;
  __syncthreads();
  for (int iter = 0; iter <= n; ++iter) {
    int best = lab[j];
    for (int w = 0; w < OA_W; ++w)
      for (unsigned b = m[w]; b; b &= b - 1u) best = min(best, lab[w * 32 + __ffs(b) - 1]);
    const int less = best < lab[j];
    const int again = __syncthreads_or(less);   // every neighbour is read before a label changes
    if (less) lab[j] = best;
    __syncthreads();
    if (!again) break;
  }
}

// Each cluster of 2..CL_MAX columns is diagonalised exactly: U, w = eig(P^H S_c P),
// P = I + R_c / 2, by one warp: Jacobi rounds of up to four disjoint pairs, a lane per
// pair for the angles and per pair and element for the rotations. The warp of a cluster
// is that of its smallest column, four columns per CTA.
constexpr int CLU_WARPS = EIG_NMAX / 32;
__global__ void __launch_bounds__(EIG_NMAX)
k_oa_cluster(OaArgs o) {
  __shared__ int lab[EIG_NMAX];
  __shared__ cplx sa[CLU_WARPS][CL_MAX][CL_MAX], su[CLU_WARPS][CL_MAX][CL_MAX], st[CLU_WARPS][CL_MAX][CL_MAX];
  __shared__ int smem_mem[CLU_WARPS][CL_MAX];
  const int n = o.n, lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  oa_labels(o.mask, n, lab);
  const int i = blockIdx.x * CLU_WARPS + wid;
  int sc = 0;                           // the size of the cluster that starts at column i
  if (i < n && lab[i] == i)
    for (int w = 0; w < OA_W; ++w) {
      const int j = w * 32 + lane, in = j < n && lab[j] == i;
      const unsigned bits = __ballot_sync(0xffffffffu, in);
      const int at = sc + __popc(bits & ((1u << lane) - 1u));
      if (in && at < CL_MAX) smem_mem[wid][at] = j;
      sc += __popc(bits);
    }
  if (i < n && lane == 0) o.label[i] = lab[i];
  if (blockIdx.x == 0) {
    int big = 0;
    for (int j = lane; j < n && wid == 0; j += 32) {
      if (lab[j] != j) continue;
      int cnt = 0;
      for (int k = j; k < n; ++k) cnt += (lab[k] == j);
      big += cnt > CL_MAX;
    }
    for (int off = 16; off > 0; off >>= 1) big += __shfl_down_sync(0xffffffffu, big, off);
    if (threadIdx.x == 0) o.stat[1] = (double)big;
  }
  __syncwarp();
  if (sc == 0) return;
  if (sc == 1 || sc > CL_MAX) {         // a wide cluster keeps its columns as they are
    for (int j = i + lane; j < n; j += 32)
      if (lab[j] == i) o.lam[j] = o.rq[j];
    return;
  }
  cplx(*a)[CL_MAX] = sa[wid], (*u)[CL_MAX] = su[wid], (*t)[CL_MAX] = st[wid];
  const int *mi = smem_mem[wid];
  // t = S_c P, a = P^H t with P = I + R_c / 2 (R = I - H)
  for (int e = lane; e < sc * sc; e += 32) {
    const int r = e / sc, c = e % sc;
    cplx acc = cmake(0.0, 0.0);
    for (int l = 0; l < sc; ++l) {
      const cplx hl = herm_at(o.H, n, mi[l], mi[c]);
      const cplx p = cmake((l == c ? 1.5 : 0.0) - 0.5 * hl.x, -0.5 * hl.y);
      acc = cadd(acc, cmul(herm_at(o.S, n, mi[r], mi[l]), p));
    }
    t[r][c] = acc;
  }
  __syncwarp();
  for (int e = lane; e < sc * sc; e += 32) {
    const int r = e / sc, c = e % sc;
    cplx acc = cmake(0.0, 0.0);
    for (int l = 0; l < sc; ++l) {
      const cplx hl = herm_at(o.H, n, mi[l], mi[r]);
      const cplx pc = cmake((l == r ? 1.5 : 0.0) - 0.5 * hl.x, 0.5 * hl.y);   // conj(P[l][r])
      acc = cadd(acc, cmul(pc, t[l][c]));
    }
    a[r][c] = acc;
    u[r][c] = cmake(r == c ? 1.0 : 0.0, 0.0);
  }
  __syncwarp();
  for (int e = lane; e < sc * sc; e += 32) {   // exact Hermitian symmetry for the Jacobi sweeps
    const int r = e / sc, c = e % sc;
    if (r >= c) continue;
    const cplx m = cmake(0.5 * (a[r][c].x + a[c][r].x), 0.5 * (a[r][c].y - a[c][r].y));
    a[r][c] = m;
    a[c][r] = cconj(m);
  }
  __syncwarp();
  const int np = sc + (sc & 1), pairs = np / 2, m = np - 1;
  const int k = lane / CL_MAX, x = lane % CL_MAX;   // pair and element of this lane
  for (int sweep = 0; sweep < 12; ++sweep) {
    double off = 0.0, dia = 0.0;
    for (int e = lane; e < sc * sc; e += 32) {
      const cplx v = a[e / sc][e % sc];
      const double m2 = v.x * v.x + v.y * v.y;
      if (e / sc == e % sc) dia += m2; else off += m2;
    }
    for (int s = 16; s > 0; s >>= 1) {
      off += __shfl_xor_sync(0xffffffffu, off, s);
      dia += __shfl_xor_sync(0xffffffffu, dia, s);
    }
    if (off <= 1e-32 * dia || off == 0.0) break;
    for (int step = 0; step < m; ++step) {
      const int ka = k - 1 + step, kb = np - 2 - k + step;
      const int pa = (k == 0) ? 0 : (ka < m ? ka : ka - m) + 1, pb = (kb < m ? kb : kb - m) + 1;
      const int p = min(pa, pb), q = max(pa, pb);
      bool act = k < pairs && q < sc;
      double cs = 1.0, sn = 0.0;
      cplx e = cmake(1.0, 0.0);
      if (act) {
        const cplx apq = a[p][q];
        const double mag = sqrt(apq.x * apq.x + apq.y * apq.y);
        act = mag > 1e-300;
        if (act) {
          e = cmake(apq.x / mag, apq.y / mag);
          const double tau = (a[q][q].x - a[p][p].x) / (2.0 * mag);
          const double tt = (tau >= 0.0 ? 1.0 : -1.0) / (fabs(tau) + sqrt(1.0 + tau * tau));
          cs = 1.0 / sqrt(1.0 + tt * tt);
          sn = tt * cs;
        }
      }
      act = act && x < sc;
      __syncwarp();
      if (act) {   // rows p, q
        const cplx ap = a[p][x], eaq = cmul(e, a[q][x]);
        a[p][x] = cmake(cs * ap.x - sn * eaq.x, cs * ap.y - sn * eaq.y);
        a[q][x] = cmake(sn * ap.x + cs * eaq.x, sn * ap.y + cs * eaq.y);
      }
      __syncwarp();
      if (act) {   // columns p, q of a and u
        const cplx ec = cconj(e);
        const cplx xp = a[x][p], exq = cmul(ec, a[x][q]);
        a[x][p] = cmake(cs * xp.x - sn * exq.x, cs * xp.y - sn * exq.y);
        a[x][q] = cmake(sn * xp.x + cs * exq.x, sn * xp.y + cs * exq.y);
        const cplx up = u[x][p], euq = cmul(ec, u[x][q]);
        u[x][p] = cmake(cs * up.x - sn * euq.x, cs * up.y - sn * euq.y);
        u[x][q] = cmake(sn * up.x + cs * euq.x, sn * up.y + cs * euq.y);
      }
      __syncwarp();
    }
  }
  for (int e = lane; e < sc * sc; e += 32) o.U[mi[e / sc] * CL_MAX + e % sc] = u[e / sc][e % sc];
  if (lane < sc) o.lam[mi[lane]] = a[lane][lane].x;
}

// row blockIdx.x of F, its columns of each cluster of 2..CL_MAX times the cluster's U
__global__ void __launch_bounds__(EIG_NMAX)
k_oa_form(OaArgs o) {
  __shared__ double red[32];
  __shared__ cplx f[EIG_NMAX];
  __shared__ int lab[EIG_NMAX];
  const int n = o.n, i = blockIdx.x, j = threadIdx.x;
  if (j < n) lab[j] = o.label[j];
  const double lm = block_max(j < n ? fabs(o.rq[j]) : 0.0, red);
  double fr = 0.0;
  if (j < n) {
    const cplx h = herm_at(o.H, n, i, j);
    const double rx = (i == j ? 1.0 : 0.0) - h.x, ry = -h.y;
    if (i == j) {
      f[j] = cmake(1.0 + 0.5 * rx, 0.0);
    } else if (lab[i] == lab[j]) {
      f[j] = cmake(0.5 * rx, 0.5 * ry);
    } else {
      const cplx sv = herm_at(o.S, n, i, j);
      const double lj = o.rq[j], gap = lj - o.rq[i];
      const double nx = sv.x + lj * rx, ny = sv.y + lj * ry;
      f[j] = cmake(nx / gap, ny / gap);
      fr = fmax(fr, (sqrt(nx * nx + ny * ny) - 1e-14 * lm) / fabs(gap));
    }
  }
  fr = block_max(fr, red);              // at least 0: its bits order like the number
  if (j == 0) atomicMax((unsigned long long *)o.stat, (unsigned long long)__double_as_longlong(fr));
  if (j >= n) return;
  const int root = lab[j];
  int sc = 0, pos = 0;
  for (int k = root; k < n; ++k) {
    const int in = lab[k] == root;
    pos += in && k < j;
    sc += in;
  }
  cplx r = f[j];
  if (sc >= 2 && sc <= CL_MAX) {
    r = cmake(0.0, 0.0);
    for (int k = root; k < n; ++k)
      if (lab[k] == root) r = cadd(r, cmul(f[k], o.U[k * CL_MAX + pos]));
  }
  o.F[(int64_t)i * n + j] = r;
}

// eigenvalues lam + shift sorted ascending into w, the columns of X likewise into V (ldv)
__global__ void k_sort_out(const double *lam, const double *shift, const cplx *X, int n, double *w, cplx *V,
                           int ldv) {
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    const double di = lam[i];
    int rank = 0;
    for (int j = 0; j < n; ++j) {
      const double dj = lam[j];
      if (dj < di || (dj == di && j < i)) ++rank;
    }
    w[rank] = di + *shift;
    for (int r = 0; r < n; ++r) V[(int64_t)r * ldv + rank] = X[(int64_t)r * n + i];
  }
}

// *out = max |H - I| (H n x n)
__global__ void k_orth_err(const cplx *__restrict__ H, int n, double *out) {
  __shared__ double red[32];
  double m = 0.0;
  for (int idx = threadIdx.x; idx < n * n; idx += blockDim.x) {
    const int i = idx / n, j = idx % n;
    const cplx h = H[idx];
    m = fmax(m, fmax(fabs(h.x - (i == j ? 1.0 : 0.0)), fabs(h.y)));
  }
  m = block_max(m, red);
  if (threadIdx.x == 0) *out = m;
}

__global__ void k_copy_square(const cplx *__restrict__ A, int n, int lda, cplx *B) {
  for (int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; idx < (int64_t)n * n;
       idx += (int64_t)gridDim.x * blockDim.x)
    B[idx] = A[(idx / n) * lda + idx % n];
}

constexpr size_t kJacobi32Smem = 200 * 1024;

}  // namespace

namespace {
thread_local int last_steps_ = 0;
}

int eigh_refined_last_steps() { return last_steps_; }

bool eigh_refined_fits(int n) { return n >= 1 && n <= EIG_NMAX; }

void eigh_refined(Exec &ex, const cplx *A, int n, int lda, double *w, cplx *V, int ldv, int nsteps) {
  if (n <= 0) return;
  ADC_REQUIRE(eigh_refined_fits(n), ADC_ERR_UNSUPPORTED, "eigh_refined: matrix too large");
  const int64_t nn = (int64_t)n * n;
  // the FP32 eigenvector work array in shared memory when both (padded) matrices fit
  const size_t mat = (size_t)n * (n + 1) * sizeof(float2);
  size_t smem = jacobi32_head_bytes(n) + mat;
  DBuf vg;
  if (smem + mat <= kJacobi32Smem) smem += mat;
  else vg = DBuf(ex, mat);
  set_smem_limit((const void *)k_jacobi32, (int)kJacobi32Smem);
  set_smem_limit((const void *)k_small_gemm, 64 * 1024);
  DBuf X0 = cbuf(ex, nn), X1 = cbuf(ex, nn), T = cbuf(ex, nn), H = cbuf(ex, nn), S = cbuf(ex, nn), F = cbuf(ex, nn);
  DBuf lam(ex, n * sizeof(double)), sc(ex, 4 * sizeof(double)), lab(ex, n * sizeof(int));
  DBuf oas(ex, (EIG_NMAX + 2 * OA_PARTS) * sizeof(double) + EIG_NMAX * OA_W * sizeof(unsigned));
  DBuf U = cbuf(ex, (int64_t)EIG_NMAX * CL_MAX);
  k_jacobi32<<<1, 1024, smem, ex.stream>>>(A, n, lda, X0.c(), sc.d(), 30, (float2 *)vg.p);
  ADC_CHECK_LAUNCH();
  const int gt = (n + SG_T - 1) / SG_T;
  const size_t gs = 2 * (size_t)SG_T * n * sizeof(cplx);
  auto product = [&](const SgArgs &g0, const SgArgs *g1) {
    k_small_gemm<<<dim3(gt, gt, g1 ? 2 : 1), SG_THREADS, gs, ex.stream>>>(g0, g1 ? *g1 : g0, n);
    ADC_CHECK_LAUNCH();
  };
  double *part = oas.d() + EIG_NMAX;
  OaArgs oa{H.c(), S.c(), n, oas.d(), lam.d(), part, (unsigned *)(part + 2 * OA_PARTS), U.c(), (int *)lab.p,
            sc.d() + 1, F.c()};
  cplx *X = X0.c(), *Xn = X1.c();
  bool ok = false;
  for (int it = 0; it < nsteps + 3; ++it) {
    // T = (A - shift) X and H = X^H X, then S = X^H T
    const SgArgs gH{X, n, 1, nullptr, X, H.c(), 1};
    product(SgArgs{A, lda, 0, sc.d(), X, T.c(), 0}, &gH);
    product(SgArgs{X, n, 1, nullptr, T.c(), S.c(), 1}, nullptr);
    k_oa_norms<<<n, EIG_NMAX, 0, ex.stream>>>(oa);
    ADC_CHECK_LAUNCH();
    k_oa_couple<<<n, EIG_NMAX, 0, ex.stream>>>(oa);
    ADC_CHECK_LAUNCH();
    k_oa_cluster<<<(n + CLU_WARPS - 1) / CLU_WARPS, EIG_NMAX, 0, ex.stream>>>(oa);
    ADC_CHECK_LAUNCH();
    k_oa_form<<<n, EIG_NMAX, 0, ex.stream>>>(oa);
    ADC_CHECK_LAUNCH();
    // X <- X F, F = (I + correction) blockdiag(U)
    product(SgArgs{X, n, 0, nullptr, F.c(), Xn, 0}, nullptr);
    std::swap(X, Xn);
    if (it + 1 >= nsteps) {
      // orthonormality of the updated vectors
      product(SgArgs{X, n, 1, nullptr, X, H.c(), 1}, nullptr);
      k_orth_err<<<1, 1024, 0, ex.stream>>>(H.c(), n, sc.d() + 3);
      ADC_CHECK_LAUNCH();
      double st[3];
      ADC_CUDA(cudaMemcpyAsync(st, sc.d() + 1, sizeof(st), cudaMemcpyDeviceToHost, ex.stream));
      ex.sync();
      last_steps_ = it + 1;
      if (st[0] <= 1e-8 && st[1] == 0.0 && st[2] <= OA_ORTH) { ok = true; break; }
    }
  }
  if (ok) {
    // eigenvalues: Rayleigh quotients of the vectors before the last update
    // (exact to the square of their error), exact ones within clusters
    k_sort_out<<<1, 256, 0, ex.stream>>>(lam.d(), sc.d(), X, n, w, V, ldv);
    ADC_CHECK_LAUNCH();
    return;
  }
  last_steps_ = -1;
  // a cluster too wide for the exact step, or no convergence: FP64 Jacobi
  k_copy_square<<<(int)std::min<int64_t>((nn + 255) / 256, 1024), 256, 0, ex.stream>>>(A, n, lda, T.c());
  ADC_CHECK_LAUNCH();
  jacobi_eigh(ex, T.c(), n, n, w, V, ldv, (int *)lab.p);
}

void jacobi_eigh(Exec &ex, cplx *A, int n, int lda, double *w, cplx *V, int ldv, int *info_dev) {
  if (n <= 0) return;
  ADC_REQUIRE(n <= 2048, ADC_ERR_UNSUPPORTED, "jacobi_eigh: matrix larger than 2048");
  DBuf work = cbuf(ex, (int64_t)n * n);
  int np = n + (n & 1), npairs = np / 2;
  size_t smem = (size_t)npairs * 4 * sizeof(double) + (size_t)(2 * npairs + 2) * sizeof(int) +
                64 * sizeof(double);
  constexpr size_t kMaxSmem = 200 * 1024;
  const size_t mats = 16 + 2 * (size_t)n * n * sizeof(cplx);
  const int in_smem = (smem + mats <= kMaxSmem) ? 1 : 0;
  if (in_smem) smem += mats;
  set_smem_limit((const void *)k_jacobi, (int)kMaxSmem);
  k_jacobi<<<1, 1024, smem, ex.stream>>>(A, n, lda, work.c(), w, V, ldv, info_dev, 40, 1e-14, in_smem);
  ADC_CHECK_LAUNCH();
}

}  // namespace adc
