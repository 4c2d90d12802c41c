// Cholesky QR of B^H for the mixed form (sm_103a): the QR factorisation the
// small-B SVD of Section IV's step ii starts from (B^H = Qb Rb, then the
// one-sided Jacobi SVD of Rb^H), for well-conditioned B.
//
// CholeskyQR2 (Yamamoto, Nakatsukasa, Yanagisawa, Fukaya, ETNA 44, 2015):
//   G1 = B B^H = R1^H R1,  Q1 = B^H R1^-1,
//   G2 = Q1^H Q1 = R2^H R2, Qb = Q1 R2^-1,
// with the Gram matrices and the triangular products FP64-accurate (on the
// tensor cores from exact digit splits, k_oz_gemm, or in double-float
// arithmetic, k_zgemm_df; stages G_G1 .. G_X) and the Cholesky
// factorisations and triangular inverses in FP64 here.  For kappa(B) below
// ~1e8 the two passes give an orthonormal Qb and a backward-stable
// factorisation (residual and orthogonality at the unit-roundoff level), so
// the singular values of Rb are those of B to ~eps ||B||.  Rb^H is formed as
// X = B Qb.  An instance whose first Gram matrix is too ill-conditioned for
// that (a Cholesky pivot below CQ_PIVOT times the largest diagonal entry,
// i.e. kappa(B) above ~1e5) is flagged (Dims::qflag) and factored by the
// Householder QR instead; its Cholesky output is replaced by the identity so
// that the products in between stay finite.
#include <cuda_runtime.h>
#include <math.h>

#include "dfsplit.cuh"
#include "internal.cuh"
#include "mixed.cuh"
#include "once.cuh"
#include "profiler.cuh"

namespace tg {

static const double CQ_PIVOT = 1e-10;
// the same bound for the scaled Gram matrix of the digit-split form (2^-30: kappa(B S) ~ 3e4)
static const float CQ_MIN_PIVOT = 9.3132257461547852e-10f;

// Cholesky G = R^H R of the l x l Hermitian matrix in P.R (upper triangle,
// column-major, in place), then J = R^-1 (upper triangular, zero below).  One
// CTA per instance.  pass 0 sets dims[p].qflag to 0 or 1; pass 1 skips the
// instances already flagged and flags those whose second Gram fails.
__global__ void __launch_bounds__(256) k_chol_inv(Dims* dims, const ProbPtr* __restrict__ ptrs, int pass) {
  __shared__ double red[32];
  __shared__ double s_inv;
  __shared__ int s_fail;
  const int p = blockIdx.x;
  const Dims D = dims[p];
  if (!D.active) return;
  if (pass == 1 && D.qflag) return;
  const ProbPtr P = ptrs[p];
  const int L = D.l, tid = threadIdx.x;
  cplx* G = P.R;
  cplx* J = P.J;
  double dm = 0.0;
  for (int j = tid; j < L; j += blockDim.x) dm = fmax(dm, G[(size_t)j * L + j].x);
  // block maximum through the sum helper's pattern
  {
    const int lane = tid & 31, warp = tid >> 5, nw = (blockDim.x + 31) >> 5;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) dm = fmax(dm, __shfl_xor_sync(0xffffffffu, dm, o));
    if (lane == 0) red[warp] = dm;
    __syncthreads();
    if (tid == 0) {
      double m = 0.0;
      for (int w = 0; w < nw; ++w) m = fmax(m, red[w]);
      red[0] = m;
      s_fail = !(m > 0.0) || !isfinite(m);
    }
    __syncthreads();
    dm = red[0];
  }
  for (int j = 0; j < L && !s_fail; ++j) {
    if (tid == 0) {
      const double d = G[(size_t)j * L + j].x;
      if (!(d > CQ_PIVOT * dm) || !isfinite(d)) {
        s_fail = 1;
      } else {
        const double r = sqrt(d);
        G[(size_t)j * L + j] = cmk(r, 0.0);
        s_inv = 1.0 / r;
      }
    }
    __syncthreads();
    if (s_fail) break;
    const double inv = s_inv;
    for (int c = j + 1 + tid; c < L; c += blockDim.x) G[(size_t)c * L + j] = cscale(G[(size_t)c * L + j], inv);
    __syncthreads();
    // trailing update of the upper triangle: G[c1][c2] -= conj(R[j][c1]) R[j][c2], j < c1 <= c2
    const int w = L - j - 1;
    for (int e = tid; e < w * w; e += blockDim.x) {
      const int c1 = j + 1 + e % w, c2 = j + 1 + e / w;
      if (c1 > c2) continue;
      const cplx a = G[(size_t)c1 * L + j], b = G[(size_t)c2 * L + j];
      cplx& g = G[(size_t)c2 * L + c1];
      g.x -= a.x * b.x + a.y * b.y;
      g.y -= a.x * b.y - a.y * b.x;
    }
    __syncthreads();
  }
  const int fail = s_fail;
  if (tid == 0) dims[p].qflag = fail ? 1 : (pass == 0 ? 0 : D.qflag);
  if (fail) {  // identity factor: the products in between stay finite
    for (int e = tid; e < L * L; e += blockDim.x) J[e] = cmk((e / L) == (e % L) ? 1.0 : 0.0, 0.0);
    return;
  }
  // J = R^-1 by back substitution, one column per thread: R x = e_c
  for (int c = tid; c < L; c += blockDim.x) {
    cplx* x = J + (size_t)c * L;
    for (int i = c + 1; i < L; ++i) x[i] = cmk(0.0, 0.0);
    for (int i = c; i >= 0; --i) {
      cplx s = cmk(i == c ? 1.0 : 0.0, 0.0);
      for (int k = i + 1; k <= c; ++k) {
        const cplx r = G[(size_t)k * L + i], v = x[k];
        s.x -= r.x * v.x - r.y * v.y;
        s.y -= r.x * v.y + r.y * v.x;
      }
      const double rii = G[(size_t)i * L + i].x;  // real and positive
      x[i] = cscale(s, 1.0 / rii);
    }
  }
}

// The same factorisation in double-float arithmetic (FP32 pairs, 2^-48;
// the FP32 pipe runs 64x the FP64 one) with the Gram's upper triangle packed
// in shared memory (element (r, c), r <= c, at c (c + 1) / 2 + r) for
// l <= CS_MAXL, then R^-1 in place, column by column (R X = I):
//   X[j][j] = 1 / R[j][j],  X[0:j, j] = -X[j][j] X[0:j, 0:j] R[0:j, j],
// the leading block X[0:j, 0:j] being the columns already inverted; each
// column's j dot products run on the threads (row r: sum over k = r .. j-1),
// into scratch first (they read the column they replace).  The trailing
// updates of the factorisation enumerate the packed pairs c1 <= c2 directly,
// so every lane does work.  G is scaled by a power of four first, so that its
// largest diagonal entry lies in [0.5, 4), and R^-1 scaled back.
enum { CS_THREADS = 256, CS_MAXL = 160 };

__host__ __device__ inline size_t cs_smem_bytes(int L) { return ((size_t)L * (L + 1) / 2 + L) * sizeof(cplx); }

__device__ __forceinline__ int cs_at(int r, int c) { return c * (c + 1) / 2 + r; }

// (a, b) with a <= b from the packed index e = b (b + 1) / 2 + a
__device__ __forceinline__ void cs_pair(int e, int& a, int& b) {
  int c = (int)((sqrtf(8.0f * (float)e + 1.0f) - 1.0f) * 0.5f);
  if ((c + 1) * (c + 2) / 2 <= e) ++c;
  if (c * (c + 1) / 2 > e) --c;
  b = c;
  a = e - c * (c + 1) / 2;
}

// Complex double-float entry: (Re hi, Re lo, Im hi, Im lo).
__device__ __forceinline__ float4 cs_split(cplx v) {
  float4 d;
  split_bits(v.x, d.x, d.y);
  split_bits(v.y, d.z, d.w);
  return d;
}

__global__ void __launch_bounds__(CS_THREADS) k_chol_inv_sm(Dims* dims, const ProbPtr* __restrict__ ptrs, int pass) {
  extern __shared__ __align__(16) unsigned char cs_raw[];
  __shared__ double red[32];
  __shared__ float2 s_inv;
  __shared__ int s_fail;
  const int p = blockIdx.x;
  const Dims D = dims[p];
  if (!D.active) return;
  if (pass == 1 && D.qflag) return;
  const ProbPtr P = ptrs[p];
  const int L = D.l, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = CS_THREADS / 32;
  float4* T = reinterpret_cast<float4*>(cs_raw);
  float4* tmp = T + (size_t)L * (L + 1) / 2;  // L
  const cplx* G = P.R;
  cplx* J = P.J;
  // the largest diagonal entry, then G scaled by 2^-2s (exact) to bring it
  // into [0.5, 4): FP32's range holds the factor, R^-1 is scaled back by 2^s
  double dm = 0.0;
  for (int c = tid; c < L; c += CS_THREADS) dm = fmax(dm, G[(size_t)c * L + c].x);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) dm = fmax(dm, __shfl_xor_sync(0xffffffffu, dm, o));
  if (lane == 0) red[warp] = dm;
  __syncthreads();
  if (tid == 0) {
    double m = 0.0;
    for (int w = 0; w < nw; ++w) m = fmax(m, red[w]);
    red[0] = m;
    s_fail = !(m > 0.0) || !isfinite(m);
  }
  __syncthreads();
  dm = red[0];
  int ex = 0;
  if (!s_fail) (void)frexp(dm, &ex);  // dm = f 2^ex, f in [0.5, 1)
  const int sh = ex >> 1;             // scale G by 2^-2 sh
  const double gsc = ldexp(1.0, -2 * sh);
  for (int e = tid; e < L * L; e += CS_THREADS) {
    const int r = e % L, c = e / L;
    if (r <= c) T[cs_at(r, c)] = cs_split(cscale(G[(size_t)c * L + r], gsc));
  }
  const float piv = (float)(CQ_PIVOT * dm * gsc);
  __syncthreads();
  for (int j = 0; j < L && !s_fail; ++j) {
    if (tid == 0) {
      const float4 dd = T[cs_at(j, j)];
      const dfl d{dd.x, dd.y};
      if (!(d.h > piv) || !isfinite(d.h)) {
        s_fail = 1;
      } else {
        const dfl r = dsqrt(d);
        const dfl inv = drecip(r);
        T[cs_at(j, j)] = make_float4(r.h, r.l, 0.f, 0.f);
        s_inv = make_float2(inv.h, inv.l);
      }
    }
    __syncthreads();
    if (s_fail) break;
    const dfl inv{s_inv.x, s_inv.y};
    for (int c = j + 1 + tid; c < L; c += CS_THREADS) {
      const float4 v = T[cs_at(j, c)];
      const dfl re = dmul(dfl{v.x, v.y}, inv), im = dmul(dfl{v.z, v.w}, inv);
      T[cs_at(j, c)] = make_float4(re.h, re.l, im.h, im.l);
    }
    __syncthreads();
    // G[c1][c2] -= conj(R[j][c1]) R[j][c2], j < c1 <= c2: the packed pairs of the trailing block
    const int w = L - j - 1, j1 = j + 1;
    for (int e = tid; e < w * (w + 1) / 2; e += CS_THREADS) {
      int a, b;
      cs_pair(e, a, b);
      const int c1 = j1 + a, c2 = j1 + b;
      const float4 x = T[cs_at(j, c1)], y = T[cs_at(j, c2)];
      float4& g = T[cs_at(c1, c2)];
      // Re -= xr yr + xi yi, Im -= xr yi - xi yr
      float rh = g.x, rl = g.y, ih = g.z, il = g.w;
      dfx_dd(rh, rl, -x.x, -x.y, y.x, y.y);
      dfx_dd(rh, rl, -x.z, -x.w, y.z, y.w);
      dfx_dd(ih, il, -x.x, -x.y, y.z, y.w);
      dfx_dd(ih, il, x.z, x.w, y.x, y.y);
      fast2(rh, rl);
      fast2(ih, il);
      g = make_float4(rh, rl, ih, il);
    }
    __syncthreads();
  }
  const int fail = s_fail;
  if (tid == 0) dims[p].qflag = fail ? 1 : (pass == 0 ? 0 : D.qflag);
  if (fail) {  // identity factor: the products in between stay finite
    for (int e = tid; e < L * L; e += CS_THREADS) J[e] = cmk((e / L) == (e % L) ? 1.0 : 0.0, 0.0);
    return;
  }
  // R^-1 in place
  for (int j = 0; j < L; ++j) {
    for (int r = tid; r < j; r += CS_THREADS) {
      float sh_ = 0.f, sl = 0.f, th = 0.f, tl = 0.f;  // Re, Im of sum_k X[r][k] R[k][j]
      for (int k = r; k < j; ++k) {
        const float4 x = T[cs_at(r, k)], u = T[cs_at(k, j)];
        dfx_dd(sh_, sl, x.x, x.y, u.x, u.y);
        dfx_dd(sh_, sl, -x.z, -x.w, u.z, u.w);
        dfx_dd(th, tl, x.x, x.y, u.z, u.w);
        dfx_dd(th, tl, x.z, x.w, u.x, u.y);
      }
      fast2(sh_, sl);
      fast2(th, tl);
      tmp[r] = make_float4(sh_, sl, th, tl);
    }
    __syncthreads();
    const float4 djj = T[cs_at(j, j)];
    const dfl dj = drecip(dfl{djj.x, djj.y});
    for (int r = tid; r <= j; r += CS_THREADS) {
      if (r == j) {
        T[cs_at(j, j)] = make_float4(dj.h, dj.l, 0.f, 0.f);
      } else {
        const float4 v = tmp[r];
        const dfl re = dmul(dfl{v.x, v.y}, dneg(dj)), im = dmul(dfl{v.z, v.w}, dneg(dj));
        T[cs_at(r, j)] = make_float4(re.h, re.l, im.h, im.l);
      }
    }
    __syncthreads();
  }
  const double back = ldexp(1.0, -sh);  // R^-1 of the unscaled G = 2^-s R'^-1
  for (int e = tid; e < L * L; e += CS_THREADS) {
    const int r = e % L, c = e / L;
    cplx v = cmk(0.0, 0.0);
    if (r <= c) {
      const float4 t = T[cs_at(r, c)];
      v = cmk(((double)t.x + (double)t.y) * back, ((double)t.z + (double)t.w) * back);
    }
    J[e] = v;
  }
}

// the kernel of the digit-split form below
template <bool SM>
__global__ void k_chol_eq(Dims* dims, const ProbPtr* __restrict__ ptrs, int pass, int passes, float min_pivot,
                          float again, int cond, int f32);

static cudaError_t lowdin_prepare();

cudaError_t cholqr_prepare() {
  static DeviceOnce once;
  return once([] {
    const int sm = (int)cs_smem_bytes(CS_MAXL);
    cudaError_t e = cudaFuncSetAttribute(k_chol_inv_sm, cudaFuncAttributeMaxDynamicSharedMemorySize, sm);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_chol_eq<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, sm);
    if (e == cudaSuccess) e = lowdin_prepare();
    if (e == cudaSuccess) e = qr_small_prepare();
    if (e == cudaSuccess) e = jac_pre_prepare();
    return e;
  });
}

static cudaError_t chol_inv(Dims* dims, const ProbPtr* ptrs, int batch, int lcap, int pass, cudaStream_t st) {
  ProfScope ps("k_chol_inv", st);
  if (lcap <= CS_MAXL) {
    const cudaError_t e = cholqr_prepare();
    if (e != cudaSuccess) return e;
    k_chol_inv_sm<<<batch, CS_THREADS, cs_smem_bytes(lcap), st>>>(dims, ptrs, pass);
  } else {
    k_chol_inv<<<batch, 256, 0, st>>>(dims, ptrs, pass);
  }
  return cudaGetLastError();
}

#define CQ_TRY(x)                     \
  do {                                \
    cudaError_t e_ = (x);             \
    if (e_ != cudaSuccess) return e_; \
  } while (0)

cudaError_t run_cholqr_bh(Dims* dims, const ProbPtr* ptrs, int batch, const Caps& cap, cudaStream_t st,
                          const OzScratch* oz, int* err, bool phases) {
  if (oz) {
    CQ_TRY(run_cholqr(1, 2, phases ? CQ_PHASES : CQ_LOWDIN, CQ_MIN_PIVOT, dims, ptrs, batch, cap, *oz, batch, 0, err, st));
    CQ_TRY(launch_oz_stage(G_X, dims, ptrs, batch, cap, *oz, err, st, DPC_OK));  // X = B Qb = Rb^H
    return launch_qr_rest(QR_BH, dims, ptrs, batch, cap, st, QRS_CF, true);
  }
  auto gemm = [&](int stage) { return launch_zgemm_df(stage, dims, ptrs, batch, cap, st); };
  CQ_TRY(gemm(G_G1));                          // G1 = B B^H
  CQ_TRY(chol_inv(dims, ptrs, batch, cap.l, 0, st));  // R1, J = R1^-1
  CQ_TRY(gemm(G_Q1));                          // Q1 = B^H R1^-1
  CQ_TRY(gemm(G_G2));                          // G2 = Q1^H Q1
  CQ_TRY(chol_inv(dims, ptrs, batch, cap.l, 1, st));  // R2, J = R2^-1
  CQ_TRY(gemm(G_QB));                          // Qb = Q1 R2^-1
  CQ_TRY(gemm(G_X));                           // X = B Qb = Rb^H
  // ill-conditioned instances: Householder QR of B^H (overwrites X and Qb)
  return launch_qr(QR_BH, dims, ptrs, batch, cap, st, QRS_QFLAG);
}

// ---------------------------------------------------------------------------
// Cholesky QR from digit-split products: Y into Q (m rows), or Yt into Qt (n).
//
// One pass is G = X^H X (56-bit digit products), the Cholesky factor R of the
// scaled S G S and its inverse in double-float arithmetic (k_chol_eq), and
// Q = (X S) R^-1 (digit products), with S the powers of two that bring the
// columns of X to norms in [1, 2).  The scaling takes out the grading of the
// columns that a power round leaves (Y = A Q~ with Q~ near the singular
// vectors: kappa(Y) up to 1/eps, kappa(Y S) of 3 to 1000, measured on CPU
// emulations of decaying spectra down to 1e-16), so one pass is enough there.
// Y0 = A Omega is as ill-conditioned as A itself: a pivot below CE_PIVOT adds
// the shift CE_SHIFT to the diagonal and asks for another pass (shifted
// Cholesky QR: Fukaya, Kannan, Nakatsukasa, Yamamoto, Yanagisawa, SIAM J. Sci.
// Comput. 42, 2020); each shifted pass brings directions of relative size
// below sqrt(CE_SHIFT) up by 1/sqrt(CE_SHIFT) ~ 2e5, so three passes take
// rounding-level directions to O(1).
//
// Q's range: the product with R^-1 is rounded to ~2^-56 kappa(X S) of a unit
// column, so the last basis before the projection and the QR of B^H ask for
// pivots above their min_pivot (kappa ~ 100: 1e-15, Householder's level),
// and the basis is then made orthonormal to FP64 by the symmetric correction
// Q (I + E)^-1/2, E = Q^H Q - I formed from digits (k_lowdin64).  Problems
// that miss a bound have cf set and are left to the Householder QR.
// ---------------------------------------------------------------------------
static const float CE_PIVOT = 5.8207660913467407e-11f;  // 2^-34: above the double-float rounding of a pivot
static const float CE_SHIFT = 2.9103830456733704e-11f;  // 2^-35
static const float CE_AGAIN = 1.4901161193847656e-08f;  // 2^-26: below it another pass, where one is left
static const float CE_AGAIN_LD = 6.103515625e-05f;      // 2^-14: the same before the symmetric correction

// (k_chol_eq: twice the warps from CE_WIDE columns on, whose updates have work for them)
enum { CE_THREADS = 512, CE_THREADS_BIG = 1024, CE_WIDE = 64, CE_MAXL = 512 };
static int ce_threads(int l) { return l > CE_WIDE ? CE_THREADS_BIG : CE_THREADS; }
static const float CE_F32_LAST = 16.f, CE_F32_MID = 1e4f;  // bounds of the FP32 form's R^-1 column sums
enum { CE_F32_EXP = 96 };  // column norms 2^+-96 leave S R^-1 inside FP32's range

// x 2^k by the exponent bits (x = 0 and results below the normal range: 0)
__device__ __forceinline__ double ce_scale(double x, int k) {
  const long long u = __double_as_longlong(x);
  const int e = (int)((u >> 52) & 0x7FF) + k;
  return (((u >> 52) & 0x7FF) == 0 || e <= 0) ? 0.0 : __longlong_as_double(u + ((long long)k << 52));
}

__device__ __forceinline__ bool ce_takes(const Dims& D, int pass, int cond) {
  if (!D.active) return false;
  if ((cond & DPC_QFLAG) && !D.qflag) return false;
  if ((cond & DPC_DIG) && !D.dig) return false;
  if ((cond & DPC_WIDE) && D.l < DP_WIDE_L) return false;
  return pass == 0 || (D.cq >= pass && !D.cf);
}

// S, R and R^-1 of the Gram matrix in P.R (full, column-major): sigma = S,
// J = R^-1 (upper triangular, zero below).  The triangle lives packed in
// shared memory (SM), or in place in P.R's upper half (the lower half keeps G
// for a second attempt with the shift).
template <bool SM>
__global__ void __launch_bounds__(CE_THREADS_BIG) k_chol_eq(Dims* dims, const ProbPtr* __restrict__ ptrs, int pass,
                                                        int passes, float min_pivot, float again, int cond,
                                                        int f32) {
  extern __shared__ __align__(16) unsigned char ce_raw[];
  __shared__ double s_diag[CE_MAXL];
  __shared__ int s_exp[CE_MAXL];
  __shared__ float2 s_inv;
  __shared__ int s_state;  // 0 factored, 1 a pivot below the bound, 2 not a Gram matrix
  __shared__ float s_min;
  __shared__ int s_sum;  // bits of a non-negative float
  const int p = blockIdx.x;
  const Dims D = dims[p];
  if (!ce_takes(D, pass, cond)) {
    if (f32 && pass == 0 && threadIdx.x == 0) dims[p].cf = 1;  // too narrow: Householder's
    return;
  }
  const ProbPtr P = ptrs[p];
  const int L = D.l, tid = threadIdx.x, nt = blockDim.x;
  cplx* G = P.R;
  cplx* J = P.J;
  float4* Tg = reinterpret_cast<float4*>(P.R);
  float4* Ts = reinterpret_cast<float4*>(ce_raw);
  float4* tmp = SM ? Ts + (size_t)L * (L + 1) / 2 : Ts;  // L
  auto T = [&](int r, int c) -> float4& { return SM ? Ts[cs_at(r, c)] : Tg[(size_t)c * L + r]; };
  if (tid == 0) {
    s_state = 0;
    s_sum = 0;
  }
  __syncthreads();
  for (int c = tid; c < L; c += nt) {
    const double d = G[(size_t)c * L + c].x;
    const int e = (int)(((unsigned long long)__double_as_longlong(d) >> 52) & 0x7FF);
    if (!(d > 0.0) || e == 0 || e == 0x7FF) s_state = 2;
    if (f32 && abs(e - 1023) > 2 * CE_F32_EXP) s_state = 2;
    s_diag[c] = d;
    s_exp[c] = -((e - 1023) >> 1);
  }
  __syncthreads();
  bool shifted = false;
  for (int attempt = 0; s_state != 2 && attempt < 2; ++attempt) {
    shifted = attempt == 1;
    for (int e = tid; e < L * L; e += nt) {
      const int r = e % L, c = e / L;
      if (r > c) continue;
      const int k = s_exp[r] + s_exp[c];
      cplx v;
      if (r == c) {
        v = cmk(s_diag[c], 0.0);
      } else {
        const cplx w = G[(size_t)r * L + c];  // the lower triangle: conj of (r, c)
        v = cmk(w.x, -w.y);
      }
      float4 t = cs_split(cmk(ce_scale(v.x, k), ce_scale(v.y, k)));
      if (r == c && shifted) {
        float h = t.x, l = t.y;
        two_sum(t.x, CE_SHIFT, h, l);
        l += t.y;
        fast2(h, l);
        t.x = h;
        t.y = l;
      }
      T(r, c) = t;
    }
    if (tid == 0) {
      s_state = 0;
      s_min = 4.f;
    }
    __syncthreads();
    const float bound = fmaxf(CE_PIVOT, min_pivot) * (shifted ? 0.25f : 1.f);
    for (int j = 0; j < L; ++j) {
      if (tid == 0) {
        const float4 dd = T(j, j);
        const dfl d{dd.x, dd.y};
        if (!(d.h > bound) || !isfinite(d.h)) {
          s_state = isfinite(d.h) ? 1 : 2;
        } else {
          const dfl r = dsqrt(d);
          const dfl inv = drecip(r);
          T(j, j) = make_float4(r.h, r.l, 0.f, 0.f);
          s_inv = make_float2(inv.h, inv.l);
          s_min = fminf(s_min, d.h);
        }
      }
      __syncthreads();
      if (s_state) break;
      const dfl inv{s_inv.x, s_inv.y};
      for (int c = j + 1 + tid; c < L; c += nt) {
        const float4 v = T(j, c);
        const dfl re = dmul(dfl{v.x, v.y}, inv), im = dmul(dfl{v.z, v.w}, inv);
        T(j, c) = make_float4(re.h, re.l, im.h, im.l);
      }
      __syncthreads();
      const int w = L - j - 1, j1 = j + 1;
      for (int e = tid; e < w * (w + 1) / 2; e += nt) {
        int a, b;
        cs_pair(e, a, b);
        const int c1 = j1 + a, c2 = j1 + b;
        const float4 x = T(j, c1), y = T(j, c2);
        float4& g = T(c1, c2);
        float rh = g.x, rl = g.y, ih = g.z, il = g.w;
        dfx_dd(rh, rl, -x.x, -x.y, y.x, y.y);
        dfx_dd(rh, rl, -x.z, -x.w, y.z, y.w);
        dfx_dd(ih, il, -x.x, -x.y, y.z, y.w);
        dfx_dd(ih, il, x.z, x.w, y.x, y.y);
        fast2(rh, rl);
        fast2(ih, il);
        g = make_float4(rh, rl, ih, il);
      }
      __syncthreads();
    }
    // a pivot below the bound: once more with the shift, where the caller takes one
    const bool retry = s_state == 1 && attempt == 0 && min_pivot == 0.f;
    __syncthreads();
    if (!retry) break;
  }
  const bool fail = s_state != 0 || (shifted && pass + 1 == passes);
  const bool more = !fail && (shifted || (!f32 && s_min < again && pass + 1 < passes));
  if (tid == 0) {
    dims[p].cf = fail ? 1 : 0;
    dims[p].cq = more ? pass + 1 : pass;
  }
  if (fail) {  // an identity factor: the products in between stay finite
    for (int e = tid; e < L * L; e += nt) J[e] = cmk((e / L) == (e % L) ? 1.0 : 0.0, 0.0);
    for (int c = tid; c < L; c += nt) P.sigma[c] = 1.0;
    return;
  }
  // R^-1 in place, column by column: X[0:j, j] = -X[j][j] X[0:j, 0:j] R[0:j, j].
  // Four lanes per row: the dot products of a column are up to j long.
  const int quad = tid >> 2, ql = tid & 3;
  for (int j = 0; j < L; ++j) {
    for (int r0 = 0; r0 < j; r0 += nt / 4) {
      const int r = r0 + quad;
      float sh = 0.f, sl = 0.f, th = 0.f, tl = 0.f;
      if (r < j)
        for (int k = r + ql; k < j; k += 4) {
          const float4 x = T(r, k), u = T(k, j);
          dfx_dd(sh, sl, x.x, x.y, u.x, u.y);
          dfx_dd(sh, sl, -x.z, -x.w, u.z, u.w);
          dfx_dd(th, tl, x.x, x.y, u.z, u.w);
          dfx_dd(th, tl, x.z, x.w, u.x, u.y);
        }
#pragma unroll
      for (int o = 1; o < 4; o <<= 1) {
        const dfl a = dadd(dfl{sh, sl}, dfl{__shfl_xor_sync(0xffffffffu, sh, o), __shfl_xor_sync(0xffffffffu, sl, o)});
        const dfl b = dadd(dfl{th, tl}, dfl{__shfl_xor_sync(0xffffffffu, th, o), __shfl_xor_sync(0xffffffffu, tl, o)});
        sh = a.h;
        sl = a.l;
        th = b.h;
        tl = b.l;
      }
      if (r < j && ql == 0) tmp[r] = make_float4(sh, sl, th, tl);
    }
    __syncthreads();
    const float4 djj = T(j, j);
    const dfl dj = drecip(dfl{djj.x, djj.y});
    __syncthreads();
    for (int r = tid; r <= j; r += nt) {
      if (r == j) {
        T(j, j) = make_float4(dj.h, dj.l, 0.f, 0.f);
      } else {
        const float4 v = tmp[r];
        const dfl re = dmul(dfl{v.x, v.y}, dneg(dj)), im = dmul(dfl{v.z, v.w}, dneg(dj));
        T(r, j) = make_float4(re.h, re.l, im.h, im.l);
      }
    }
    __syncthreads();
  }
  if (f32) {  // S R^-1 in FP32 (k_trmm_f32)
    float2* J32 = reinterpret_cast<float2*>(P.J);
    for (int e = tid; e < L * L; e += nt) {
      const int r = e % L, c = e / L;
      float2 v = make_float2(0.f, 0.f);
      if (r <= c) {
        const float4 t = T(r, c);
        const float s = __uint_as_float((unsigned)(127 + s_exp[r]) << 23);
        v = make_float2(t.x * s, t.z * s);
      }
      J32[e] = v;
    }
    // Column c of the product is rounded to 6e-8 of sum_r |R^-1_rc| (the
    // pivots say little about it): another pass where that is above `again`,
    // none left: given up
    float worst = 0.f;
    for (int c = tid; c < L; c += nt) {
      float sum = 0.f;
      for (int r = 0; r <= c; ++r) {
        const float4 t = T(r, c);
        sum += fabsf(t.x) + fabsf(t.z);
      }
      worst = (sum > worst || sum != sum) ? sum : worst;
    }
    if (tid < L) atomicMax(&s_sum, __float_as_int(worst) & 0x7FFFFFFF);
    __syncthreads();
    if (tid == 0 && !more && !(__int_as_float(s_sum) <= again)) {
      if (pass + 1 < passes) dims[p].cq = pass + 1;
      else dims[p].cf = 1;
    }
    return;
  }
  for (int e = tid; e < L * L; e += nt) {
    const int r = e % L, c = e / L;
    cplx v = cmk(0.0, 0.0);
    if (r <= c) {
      const float4 t = T(r, c);
      v = cmk((double)t.x + (double)t.y, (double)t.z + (double)t.w);
    }
    J[e] = v;
  }
  for (int c = tid; c < L; c += nt) P.sigma[c] = ce_scale(1.0, s_exp[c]);
}

// Column phases of the Householder QR.  The Cholesky QR has a positive
// diagonal of R; the Householder QR of this library (alpha = -e^{i arg x0}
// ||x||) multiplies column j of Q by -e^{-i phi_j}, phi_j the phase of the
// leading entry of column j when reflector j is formed.  These phases come
// from a modified LU of Q's leading l x l block (Ballard, Demmel, Grigori,
// Jacquelin, Knight, Nguyen, Solomonik, IPDPS 2014): at step j the entry
// x = M[j][j] of the Schur complement gives s = -x / |x|, M[j][j] - s is the
// pivot (of modulus at least 1) and the trailing block is eliminated as
// usual.  The singular vectors then keep the phases they have when the
// Householder QR factors the basis.  Double-float, the block in P.J; the
// phases conj(s) go to P.Jk.
__global__ void __launch_bounds__(CE_THREADS) k_hh_phase(const Dims* __restrict__ dims,
                                                         const ProbPtr* __restrict__ ptrs, int side, int cond) {
  __shared__ float4 s_col[CE_MAXL];  // the multipliers of column j
  const int p = blockIdx.x;
  const Dims D = dims[p];
  if (!ce_takes(D, 0, cond) || D.cf) return;
  const ProbPtr P = ptrs[p];
  const int L = D.l, ld = side == 0 ? D.m : D.n, tid = threadIdx.x;
  const cplx* Q = side == 0 ? P.Q : P.Qt;
  float4* M = reinterpret_cast<float4*>(P.J);  // column-major L x L
  for (int e = tid; e < L * L; e += CE_THREADS) M[e] = cs_split(Q[(size_t)(e / L) * ld + e % L]);
  __syncthreads();
  for (int j = 0; j < L; ++j) {
    const float4 x = M[(size_t)j * L + j];
    // s = -x / |x| (1 for an entry negligible against the unit column)
    const dfl a2 = dadd(dmul(dfl{x.x, x.y}, dfl{x.x, x.y}), dmul(dfl{x.z, x.w}, dfl{x.z, x.w}));
    dfl sr{-1.f, 0.f}, si{0.f, 0.f};
    if (a2.h > 1e-30f) {
      const dfl ia = drecip(dsqrt(a2));
      sr = dneg(dmul(dfl{x.x, x.y}, ia));
      si = dneg(dmul(dfl{x.z, x.w}, ia));
    }
    if (tid == 0) {
      double re = (double)sr.h + (double)sr.l, im = (double)si.h + (double)si.l;
      const double f = 1.0 / sqrt(fma(re, re, im * im));  // unit modulus to FP64
      P.Jk[j] = cmk(re * f, -im * f);
    }
    // 1 / (x - s)
    const dfl pr = dadd(dfl{x.x, x.y}, dneg(sr)), pi = dadd(dfl{x.z, x.w}, dneg(si));
    const dfl id = drecip(dadd(dmul(pr, pr), dmul(pi, pi)));
    const dfl ir = dmul(pr, id), ii = dneg(dmul(pi, id));
    for (int r = j + 1 + tid; r < L; r += CE_THREADS) {
      const float4 v = M[(size_t)j * L + r];
      const dfl a{v.x, v.y}, b{v.z, v.w};
      const dfl re = dadd(dmul(a, ir), dneg(dmul(b, ii))), im = dadd(dmul(a, ii), dmul(b, ir));
      s_col[r] = make_float4(re.h, re.l, im.h, im.l);
    }
    __syncthreads();
    const int w = L - j - 1;
    for (int e = tid; e < w * w; e += CE_THREADS) {
      const int r = j + 1 + e % w, c = j + 1 + e / w;
      const float4 u = s_col[r], v = M[(size_t)c * L + j];
      float4& g = M[(size_t)c * L + r];
      float rh = g.x, rl = g.y, ih = g.z, il = g.w;
      dfx_dd(rh, rl, -u.x, -u.y, v.x, v.y);
      dfx_dd(rh, rl, u.z, u.w, v.z, v.w);
      dfx_dd(ih, il, -u.x, -u.y, v.z, v.w);
      dfx_dd(ih, il, -u.z, -u.w, v.x, v.y);
      fast2(rh, rl);
      fast2(ih, il);
      g = make_float4(rh, rl, ih, il);
    }
    __syncthreads();
  }
}

// J = (I + E)^-1/2 = I - E/2 + 3 E^2/8 to FP64 from G = I + E in P.R, for
// l max|E| <= 3e-6 (the next term is below 1e-17); S = 1.  E^2 enters at the
// level of 1e-12 at most, so it is formed in FP32, and not at all where it is
// below FP64's resolution.  phases: column j also takes k_hh_phase's phase.
enum { LW_MAXL = 160 };
static size_t lw_smem_bytes(int l) { return l <= LW_MAXL ? sizeof(float2) * (size_t)l * l : 0; }
template <bool SVD>
__global__ void __launch_bounds__(512) k_lowdin64(Dims* dims, const ProbPtr* __restrict__ ptrs, int cond,
                                                  int phases, int cap_l) {
  extern __shared__ float2 lw_e[];
  __shared__ float red[16];
  const int p = blockIdx.x;
  const Dims D = dims[p];
  if (!ce_takes(D, 0, cond) || (SVD ? D.js != 1 : D.cf != 0)) return;
  const ProbPtr P = ptrs[p];
  const int L = D.l, tid = threadIdx.x;
  const cplx* G = SVD ? P.Y : P.R;
  cplx* T = SVD ? P.Yt : P.J;
  // SVD: |E|^2 summed (an FP32 J of l = 262 has columns off by 4e-5, whose
  // bound l max|E| says nothing), else max|E|
  float mx = 0.f;
  for (int e = tid; e < L * L; e += 512) {
    const cplx g = G[e];
    const float re = (float)((e / L == e % L) ? g.x - 1.0 : g.x), im = (float)g.y;
    if (SVD) {
      mx += fmaf(re, re, im * im);
    } else {
      const float m = fmaxf(fabsf(re), fabsf(im));
      mx = (m > mx || m != m) ? m : mx;  // NaN sticks
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const float y = __shfl_xor_sync(0xffffffffu, mx, o);
    mx = SVD ? mx + y : ((y > mx || y != y) ? y : mx);
  }
  if ((tid & 31) == 0) red[tid >> 5] = mx;
  __syncthreads();
  mx = 0.f;
  for (int w = 0; w < 16; ++w) mx = SVD ? mx + red[w] : ((red[w] > mx || red[w] != red[w]) ? red[w] : mx);
  // (an FP32 J is farther from unitary, and takes a second round: 0.3 |E|^3
  // of the first is below 3e-6, of the second below FP64)
  const bool ok = SVD ? mx <= 4e-4f : mx * (float)L <= 3e-6f;
  if (!ok && tid == 0) {
    if (SVD) dims[p].js = 0;
    else dims[p].cf = 1;
  }
  if (!SVD)
    for (int c = tid; c < L; c += 512) P.sigma[c] = 1.0;
  // E in FP32 in shared memory (a conversion is an FP64
  // instruction: made per use they were nearly all of the time, 0.71 ms for
  // 16 instances of l = 120, 0.06 ms made once)
  if (cap_l > LW_MAXL) return;  // k_lowdin64_tile does the rest
  const bool square = ok && mx > (SVD ? 1e-18f : 1e-9f);
  if (square) {
    for (int e = tid; e < L * L; e += 512) {
      const cplx g = G[e];
      lw_e[e] = make_float2((float)(e % L == e / L ? g.x - 1.0 : g.x), (float)g.y);
    }
    __syncthreads();
  }
  for (int e = tid; e < L * L; e += 512) {
    const int a = e % L, b = e / L;
    const cplx g = G[e];
    cplx t = cmk(a == b ? 1.0 : 0.0, 0.0);
    if (ok) {
      t = cmk(a == b ? 1.0 - 0.5 * (g.x - 1.0) : -0.5 * g.x, -0.5 * g.y);
      if (square) {
        float sx = 0.f, sy = 0.f;
        for (int k = 0; k < L; ++k) {
          float2 u, v;
          u = lw_e[k * L + a];
          v = lw_e[b * L + k];
          sx = fmaf(u.x, v.x, fmaf(-u.y, v.y, sx));
          sy = fmaf(u.x, v.y, fmaf(u.y, v.x, sy));
        }
        t.x += 0.375 * (double)sx;
        t.y += 0.375 * (double)sy;
      }
    }
    T[e] = phases ? cmul(t, P.Jk[b]) : t;
  }
}

// The same J for l above LW_MAXL (k_lowdin64 has checked max|E|), 32 x 32 per
// CTA: l = 262 on one CTA without the shared copy took 12 ms.
template <bool SVD>
__global__ void __launch_bounds__(256) k_lowdin64_tile(const Dims* __restrict__ dims,
                                                       const ProbPtr* __restrict__ ptrs, int cond, int phases) {
  __shared__ float2 A[32][33], Bt[32][33];  // E in FP32: [k][a], [b][k]
  const int p = blockIdx.z;
  const Dims D = dims[p];
  const int L = D.l, a0 = blockIdx.x * 32, b0 = blockIdx.y * 32;
  if (!ce_takes(D, 0, cond) || (SVD ? D.js != 1 : D.cf != 0) || a0 >= L || b0 >= L) return;
  const ProbPtr P = ptrs[p];
  const cplx* G = SVD ? P.Y : P.R;
  cplx* T = SVD ? P.Yt : P.J;
  const int lane = threadIdx.x & 31, ty = threadIdx.x >> 5;
  auto at = [&](int r, int c) {
    const cplx g = G[(size_t)c * L + r];
    return make_float2((float)(r == c ? g.x - 1.0 : g.x), (float)g.y);
  };
  float2 acc[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) acc[q] = make_float2(0.f, 0.f);
  for (int k0 = 0; k0 < L; k0 += 32) {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int y = ty + 8 * q;
      A[y][lane] = (k0 + y < L && a0 + lane < L) ? at(a0 + lane, k0 + y) : make_float2(0.f, 0.f);
      Bt[y][lane] = (b0 + y < L && k0 + lane < L) ? at(k0 + lane, b0 + y) : make_float2(0.f, 0.f);
    }
    __syncthreads();
#pragma unroll 8
    for (int k = 0; k < 32; ++k) {
      const float2 u = A[k][lane];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const float2 v = Bt[ty + 8 * q][k];
        acc[q].x = fmaf(u.x, v.x, fmaf(-u.y, v.y, acc[q].x));
        acc[q].y = fmaf(u.x, v.y, fmaf(u.y, v.x, acc[q].y));
      }
    }
    __syncthreads();
  }
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int a = a0 + lane, b = b0 + ty + 8 * q;
    if (a < L && b < L) {
      const cplx g = G[(size_t)b * L + a];
      const cplx t = cmk((a == b ? 1.0 - 0.5 * (g.x - 1.0) : -0.5 * g.x) + 0.375 * (double)acc[q].x,
                         -0.5 * g.y + 0.375 * (double)acc[q].y);
      T[(size_t)b * L + a] = phases ? cmul(t, P.Jk[b]) : t;
    }
  }
}

template <bool SVD>
static cudaError_t launch_lowdin64(Dims* dims, const ProbPtr* ptrs, int batch, int l, int cond, int phases,
                                   cudaStream_t st) {
  ProfScope ps("k_lowdin", st);
  k_lowdin64<SVD><<<batch, 512, lw_smem_bytes(l), st>>>(dims, ptrs, cond, phases, l);
  if (l > LW_MAXL) {
    const int nb = (l + 31) / 32;
    k_lowdin64_tile<SVD><<<dim3(nb, nb, batch), 256, 0, st>>>(dims, ptrs, cond, phases);
  }
  return cudaGetLastError();
}

static cudaError_t lowdin_prepare() {
  for (cudaError_t e : {cudaFuncSetAttribute(k_lowdin64<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)lw_smem_bytes(LW_MAXL)),
                        cudaFuncSetAttribute(k_lowdin64<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)lw_smem_bytes(LW_MAXL))})
    if (e != cudaSuccess) return e;
  return cudaSuccess;
}

static size_t ce_smem_bytes(int L) { return L <= CS_MAXL ? cs_smem_bytes(L) : sizeof(float4) * (size_t)L; }

cudaError_t run_cholqr(int side, int passes, int lowdin, float min_pivot, Dims* dims, const ProbPtr* ptrs, int batch,
                       const Caps& cap, const OzScratch& oz, int chunk, int cond, int* err, cudaStream_t st) {
  const float again = (lowdin & CQ_SHIFTED) ? 0.f : (lowdin ? CE_AGAIN_LD : CE_AGAIN);
  lowdin &= ~CQ_SHIFTED;
  auto prod = [&](int stage, int c) {
    return launch_oz_range(stage, dims, ptrs, batch, cap, oz, chunk, c, err, st);
  };
  CQ_TRY(cholqr_prepare());
  const int g0 = side == 0 ? G_CYG : G_CTG, q0 = side == 0 ? G_CYQ : G_CTQ;
  const int g1 = side == 0 ? G_CQG : G_CRG, q1 = side == 0 ? G_CQQ : G_CRQ;
  for (int pass = 0; pass < passes; ++pass) {
    const int in_pass = cond | (pass << DPC_PASS);
    CQ_TRY(prod(pass ? g1 : g0, in_pass | (pass ? DPC_OK : 0)));
    {
      ProfScope ps("k_chol_inv", st);
      const float mp = pass == 0 ? min_pivot : 0.f;
      if (cap.l <= CS_MAXL)
        k_chol_eq<true><<<batch, ce_threads(cap.l), ce_smem_bytes(cap.l), st>>>(dims, ptrs, pass, passes, mp, again, cond, 0);
      else
        k_chol_eq<false><<<batch, ce_threads(cap.l), ce_smem_bytes(cap.l), st>>>(dims, ptrs, pass, passes, mp, again, cond, 0);
      CQ_TRY(cudaGetLastError());
    }
    CQ_TRY(prod(pass ? q1 : q0, in_pass | DPC_OK));
  }
  if (!lowdin) return cudaSuccess;
  if (lowdin == CQ_PHASES) {
    ProfScope ps("k_hh_phase", st);
    k_hh_phase<<<batch, CE_THREADS, 0, st>>>(dims, ptrs, side, cond);
    CQ_TRY(cudaGetLastError());
  }
  CQ_TRY(prod(g1, cond | DPC_OK));
  CQ_TRY(launch_lowdin64<false>(dims, ptrs, batch, cap.l, cond, lowdin == CQ_PHASES, st));
  return prod(q1, cond | DPC_OK);
}

cudaError_t run_cholqr_f32(float2* A, float2* Q, int M, int l, int use_n, bool last, Dims* dims, const ProbPtr* ptrs,
                           int batch, const OzScratch& oz, int* err, cudaStream_t st) {
  CQ_TRY(cholqr_prepare());
  enum { PASSES = 4 };
  for (int pass = 0; pass < PASSES; ++pass) {
    const float2* X = pass ? Q : A;
    const int cond = DPC_WIDE | (pass ? (pass << DPC_PASS) | DPC_OK : 0);
    CQ_TRY(launch_oz_gram_f32(dims, ptrs, X, oz.ad, oz.as, M, l, use_n, batch, cond, err, st));
    {
      ProfScope ps("k_chol_inv", st);
      const float again = last ? CE_F32_LAST : CE_F32_MID;
      if (l <= CS_MAXL)
        k_chol_eq<true><<<batch, ce_threads(l), ce_smem_bytes(l), st>>>(dims, ptrs, pass, PASSES, 0.f, again, DPC_WIDE, 1);
      else
        k_chol_eq<false><<<batch, ce_threads(l), ce_smem_bytes(l), st>>>(dims, ptrs, pass, PASSES, 0.f, again, DPC_WIDE, 1);
      CQ_TRY(cudaGetLastError());
    }
    CQ_TRY(launch_trmm_f32(X, Q, dims, ptrs, M, l, use_n, pass, batch, st));
  }
  return cudaSuccess;
}

cudaError_t launch_lowdin_j(Dims* dims, const ProbPtr* ptrs, int batch, int l, int cond, cudaStream_t st) {
  return launch_lowdin64<true>(dims, ptrs, batch, l, cond, 0, st);
}

cudaError_t DpPath::svd() const {
  if (!dp || !jac_pre_rule(cap, dp->chunk >= batch)) return cudaSuccess;
  return run_jac_pre(const_cast<Dims*>(dims), ptrs, batch, cap, dp->oz, dp->chunk, DPC_DIG, true, dp->err, st);
}

cudaError_t DpPath::qr(int stage, int kind) const {
  if (!dp || kind == DPQ_LAST0) return launch_qr_sized(stage, dims, ptrs, batch, cap, st);
  const int side = stage == QR_Y ? 0 : 1;
  const int check = kind == DPQ_CHECK ? DPC_QFLAG : 0;
  const bool first = kind == DPQ_FIRST || kind == DPQ_FIRST_LD;
  // A middle basis is well-conditioned once its columns are scaled, unless
  // theta's rank is below l to rounding: A^H q of the directions past it is
  // what q has left of the leading singular vectors, the same direction for
  // all.  Those take shifted passes as the first basis does (one 2000 x 2000
  // of spectrum exp(-j / 2), l = 120, q = 1: 76 ms with the Householder QR on
  // one CTA instead, 19 ms so; where none needs them the launches cost 0.08 ms
  // a basis of 16 x 2000 x 120).
  const bool mid = kind == DPQ_MID;
  const int passes = first || mid ? 3 : (kind == DPQ_CHECK ? 2 : 1);
  const int lowdin = kind == DPQ_LAST ? CQ_PHASES
                     : mid            ? CQ_SHIFTED
                                      : (kind == DPQ_CHECK || kind == DPQ_FIRST_LD ? CQ_LOWDIN : 0);
  const float min_pivot = first || mid ? 0.f : (kind == DPQ_LAST ? CE_AGAIN_LD : CE_PIVOT);
  CQ_TRY(run_cholqr(side, passes, lowdin, min_pivot, const_cast<Dims*>(dims), ptrs, batch, cap, dp->oz, dp->chunk,
                    DPC_DIG | check, dp->err, st));
  if (stage == QR_BH) CQ_TRY(launch_dp_stage(G_X, *this, DPC_DIG | DPC_OK));  // X = B Qb = Rb^H
  return launch_qr_rest(stage, dims, ptrs, batch, cap, st, check ? QRS_QFLAG_REST : QRS_REST, kind == DPQ_LAST);
}

}  // namespace tg
