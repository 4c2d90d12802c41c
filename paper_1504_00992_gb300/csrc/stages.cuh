// Stage bodies of the bond update as device functions executed by a whole
// CTA: the batched kernels (one problem or tile per CTA) and the fused
// per-bond kernel (fused.cu) run the same code.  Plain FP64.
#pragma once
#include <cuda_runtime.h>
#include <math.h>

#include "internal.cuh"

namespace tg {

// ---------------------------------------------------------------------------
// Batched complex GEMM C = op(A) op(B), FP64.
// Operands are addressed by (row stride, column stride) so the same code
// serves row- and column-major buffers; loads map consecutive threads onto the
// unit-stride direction.
// ---------------------------------------------------------------------------
struct GemmOp {
  int M, N, K;
  const cplx* A; int64_t ars, acs;
  const cplx* B; int64_t brs, bcs;
  cplx* C; int64_t crs, ccs;
};

template <int STAGE>
__device__ __forceinline__ GemmOp gemm_of(const Dims& D, const ProbPtr& P) {
  GemmOp g;
  if (STAGE == G_Y0 || STAGE == G_Y) {  // Y = A Omega  /  Y = A Q~   (m x l, column-major)
    g.M = D.m; g.N = D.l; g.K = D.n;
    g.A = P.theta; g.ars = D.n; g.acs = 1;
    g.B = (STAGE == G_Y0) ? P.omega : P.Qt; g.brs = 1; g.bcs = D.n;
    g.C = P.Y; g.crs = 1; g.ccs = D.m;
  } else if (STAGE == G_YT || STAGE == G_BH) {  // Y~ = A^H Q (n x l, column-major)
    g.M = D.n; g.N = D.l; g.K = D.m;
    g.A = P.theta; g.ars = 1; g.acs = D.n;       // op(A)(r, k) = conj(A[k][r])
    g.B = P.Q; g.brs = 1; g.bcs = D.m;
    g.C = P.Yt; g.crs = 1; g.ccs = D.n;
  } else if (STAGE == G_U) {  // U = Q Jk (m x k, row-major)
    g.M = D.m; g.N = D.k; g.K = D.l;
    g.A = P.Q; g.ars = 1; g.acs = D.m;
    g.B = P.Jk; g.brs = 1; g.bcs = D.l;
    g.C = P.U; g.crs = D.k; g.ccs = 1;
  } else if (STAGE == G_V) {  // V = Qb Wk, stored conjugated as Vh (k x n, row-major)
    g.M = D.n; g.N = D.k; g.K = D.l;
    g.A = P.Qt; g.ars = 1; g.acs = D.n;
    g.B = P.Wk; g.brs = 1; g.bcs = D.l;
    g.C = P.V; g.crs = 1; g.ccs = D.n;
  } else if (STAGE == G_PR) {  // Br = A Omega_r -> columns l .. l+r-1 of Y (m x r)
    g.M = D.m; g.N = D.r; g.K = D.n;
    g.A = P.theta; g.ars = D.n; g.acs = 1;
    g.B = P.omega; g.brs = 1; g.bcs = D.n;
    g.C = P.Y + (int64_t)D.l * D.m; g.crs = 1; g.ccs = D.m;
  } else if (STAGE == G_PQ) {  // C1 = Q^H Br (l x r, column-major in R)
    g.M = D.l; g.N = D.r; g.K = D.m;
    g.A = P.Q; g.ars = D.m; g.acs = 1;          // op(A)(i, k) = conj(Q[k][i])
    g.B = P.Y + (int64_t)D.l * D.m; g.brs = 1; g.bcs = D.m;
    g.C = P.R; g.crs = 1; g.ccs = D.l;
  } else if (STAGE == G_PD) {  // Dr = Q C1 (m x r)
    g.M = D.m; g.N = D.r; g.K = D.l;
    g.A = P.Q; g.ars = 1; g.acs = D.m;
    g.B = P.R; g.brs = 1; g.bcs = D.l;
    g.C = P.Dr; g.crs = 1; g.ccs = D.m;
  } else if (STAGE == G_G1 || STAGE == G_G2 || STAGE == G_X) {
    // l x l Gram-type products with the n x l column-major B^H (Yt), Q1
    // (omega) or Qb (Qt): G1 = Yt^H Yt, G2 = omega^H omega, X = Yt^H Qt
    const cplx* L = (STAGE == G_G2) ? P.omega : P.Yt;
    const cplx* Rt = (STAGE == G_G1) ? P.Yt : (STAGE == G_G2 ? P.omega : P.Qt);
    g.M = D.l; g.N = D.l; g.K = D.n;
    g.A = L; g.ars = D.n; g.acs = 1;             // op(A)(i, k) = conj(L[k][i])
    g.B = Rt; g.brs = 1; g.bcs = D.n;
    g.C = P.R; g.crs = 1; g.ccs = D.l;
  } else if (STAGE == G_JG || STAGE == G_JT || STAGE == G_XJ || STAGE == G_XG || STAGE == G_XT) {
    const cplx* L = (STAGE == G_JG || STAGE == G_JT) ? P.J : P.R;
    const cplx* Rt = (STAGE == G_JG || STAGE == G_XJ) ? P.J : (STAGE == G_XG ? P.R : P.Yt);
    const bool gram = STAGE == G_JG || STAGE == G_XG;
    g.M = g.N = g.K = D.l;
    g.A = L; g.ars = gram ? D.l : 1; g.acs = gram ? 1 : D.l;
    g.B = Rt; g.brs = 1; g.bcs = D.l;
    g.C = gram ? P.Y : (STAGE == G_JT ? P.J : P.R); g.crs = 1; g.ccs = D.l;
  } else if (STAGE == G_CYG || STAGE == G_CQG || STAGE == G_CTG || STAGE == G_CRG) {  // X^H X of a basis
    const bool y = (STAGE == G_CYG || STAGE == G_CQG);
    const cplx* X = (STAGE == G_CYG) ? P.Y : (STAGE == G_CQG) ? P.Q : (STAGE == G_CTG) ? P.Yt : P.Qt;
    g.M = D.l; g.N = D.l; g.K = y ? D.m : D.n;
    g.A = X; g.ars = g.K; g.acs = 1;
    g.B = X; g.brs = 1; g.bcs = g.K;
    g.C = P.R; g.crs = 1; g.ccs = D.l;
  } else if (STAGE == G_CYQ || STAGE == G_CQQ || STAGE == G_CTQ || STAGE == G_CRQ) {  // (X S) J
    const bool y = (STAGE == G_CYQ || STAGE == G_CQQ);
    const cplx* X = (STAGE == G_CYQ) ? P.Y : (STAGE == G_CQQ) ? P.Q : (STAGE == G_CTQ) ? P.Yt : P.Qt;
    g.M = y ? D.m : D.n; g.N = D.l; g.K = D.l;
    g.A = X; g.ars = 1; g.acs = g.M;
    g.B = P.J; g.brs = 1; g.bcs = D.l;
    g.C = y ? P.Q : P.Qt; g.crs = 1; g.ccs = g.M;
  } else {  // G_Q1 = Yt J, G_QB = omega J: n x l times the l x l inverse factor
    g.M = D.n; g.N = D.l; g.K = D.l;
    g.A = (STAGE == G_Q1) ? P.Yt : P.omega; g.ars = 1; g.acs = D.n;
    g.B = P.J; g.brs = 1; g.bcs = D.l;
    g.C = (STAGE == G_Q1) ? P.omega : P.Qt; g.crs = 1; g.ccs = D.n;
  }
  return g;
}

template <int STAGE>
struct StageFlags {
  static constexpr bool conjA =
      (STAGE == G_YT || STAGE == G_BH || STAGE == G_PQ || STAGE == G_G1 || STAGE == G_G2 || STAGE == G_X ||
       STAGE == G_CYG || STAGE == G_CQG || STAGE == G_CTG || STAGE == G_CRG || STAGE == G_JG || STAGE == G_XG);
  // the left operand's column k is scaled by sigma[k] (a power of two)
  // (scaleB: and the right operand's row k by its inverse)
  static constexpr bool scaleB = (STAGE == G_XJ || STAGE == G_XT);
  static constexpr bool scaleA =
      (STAGE == G_CYQ || STAGE == G_CQQ || STAGE == G_CTQ || STAGE == G_CRQ || scaleB);
  static constexpr bool conjC = (STAGE == G_V);
};

enum { ZG_TK = 16 };

// Block-wide sums of the stages take RED_LANES per-thread partials (threads
// >= RED_LANES add zeros), so CTAs of 256, 512 or 1024 threads give
// bit-identical results.
enum { RED_LANES = 256 };

// One T x T output tile of op(A) op(B) for a CTA of 256 threads (S x S
// outputs each), K in slices of ZG_TK staged through shared memory As / Bs.
template <int T, int STAGE>
__device__ __forceinline__ void zgemm_tile_dev(const GemmOp& g, int tm, int tn, cplx (*As)[T + 1],
                                               cplx (*Bs)[T + 1]) {
  constexpr int TK = ZG_TK;
  constexpr int S = T / 16;  // outputs per thread along each direction
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  const bool ccol = (g.crs == 1);
  cplx acc[S][S];
#pragma unroll
  for (int i = 0; i < S; ++i)
#pragma unroll
    for (int j = 0; j < S; ++j) acc[i][j] = cmk(0.0, 0.0);

  for (int k0 = 0; k0 < g.K; k0 += TK) {
    // A tile: op(A)(tm + r, k0 + kk) -> As[kk][r]
    for (int e = tid; e < T * TK; e += 256) {
      int r, kk;
      if (g.acs == 1) { kk = e % TK; r = e / TK; } else { r = e % T; kk = e / T; }
      const int gr = tm + r, gk = k0 + kk;
      cplx v = cmk(0.0, 0.0);
      if (gr < g.M && gk < g.K) {
        v = g.A[(int64_t)gr * g.ars + (int64_t)gk * g.acs];
        if (StageFlags<STAGE>::conjA) v.y = -v.y;
      }
      As[kk][r] = v;
    }
    // B tile: B(k0 + kk, tn + c) -> Bs[kk][c]
    for (int e = tid; e < T * TK; e += 256) {
      int c, kk;
      if (g.brs == 1) { kk = e % TK; c = e / TK; } else { c = e % T; kk = e / T; }
      const int gc = tn + c, gk = k0 + kk;
      cplx v = cmk(0.0, 0.0);
      if (gc < g.N && gk < g.K) v = g.B[(int64_t)gk * g.brs + (int64_t)gc * g.bcs];
      Bs[kk][c] = v;
    }
    __syncthreads();
#pragma unroll 4
    for (int kk = 0; kk < TK; ++kk) {
      cplx a[S], b[S];
#pragma unroll
      for (int i = 0; i < S; ++i) a[i] = As[kk][(ccol ? tx : ty) + 16 * i];
#pragma unroll
      for (int j = 0; j < S; ++j) b[j] = Bs[kk][(ccol ? ty : tx) + 16 * j];
#pragma unroll
      for (int i = 0; i < S; ++i)
#pragma unroll
        for (int j = 0; j < S; ++j) cfma(acc[i][j], a[i], b[j]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < S; ++i)
#pragma unroll
    for (int j = 0; j < S; ++j) {
      const int r = tm + (ccol ? tx : ty) + 16 * i, c = tn + (ccol ? ty : tx) + 16 * j;
      if (r < g.M && c < g.N) {
        cplx v = acc[i][j];
        if (StageFlags<STAGE>::conjC) v.y = -v.y;
        g.C[(int64_t)r * g.crs + (int64_t)c * g.ccs] = v;
      }
    }
}

enum { QR_MAXL = 512 };

enum { QR_THREADS = 1024, JAC_THREADS = 512 };

// ---------------------------------------------------------------------------
// Householder QR.  FP64 runs at half a multiply-add per clock on each quarter
// of an SM: a warp's FP64 instruction takes 64 clocks there, whether the next
// one depends on it or not and however many lanes take part (measured: 65
// clocks a step for a dependent chain, 64 for eight independent ones; 128 with
// two warps on the quarter).  So what counts is the number of warp
// instructions on the fullest quarter, and for the chain of reflectors that
// its warp has a quarter for itself:
//   - warp 0 alone applies H_j to column j + 1 and forms the next reflector,
//     one row per lane at a time (qr_next: ~50 instructions for 64 rows), while
//     the others apply H_j to the columns right of it, 16 lanes per column
//     (qr_apply: ~36 instructions for two columns); one barrier per column;
//   - the others' work is dealt out to the other quarters first (qr_slot);
//   - re and im sums of an inner product share the additions of the reduction
//     (qr_csum), square roots and reciprocals are one third-order step from an
//     FP32 seed, powers of two go into the exponent bits;
//   - Q's columns are independent: one warp each, in registers.
// The sums and their order are fixed by the column's role alone, so the
// one-CTA kernel, the cluster kernel (qr_small.cu) and the fused kernel give
// the same results bit for bit.
// ---------------------------------------------------------------------------
enum { QR_G = 16 };

// sums of re and im over the G lanes of a group, to all of them
template <int G>
__device__ __forceinline__ cplx qr_csum(double re, double im, int lane, unsigned mask) {
  const bool odd = lane & 1;
  double v = odd ? im : re;
  v += __shfl_xor_sync(mask, odd ? re : im, 1);
#pragma unroll
  for (int o = G / 2; o > 1; o >>= 1) v += __shfl_xor_sync(mask, v, o);
  const double w = __shfl_xor_sync(mask, v, 1);
  return odd ? cmk(w, v) : cmk(v, w);
}
// biased exponent, and x 2^k by the exponent bits (0 where that leaves the normal range below)
__device__ __forceinline__ int qr_exp(double x) { return (int)((__double_as_longlong(x) >> 52) & 0x7FF); }
__device__ __forceinline__ double qr_scale(double x, int k) {
  const int e = qr_exp(x);
  return (e == 0 || e + k <= 0) ? 0.0 : __longlong_as_double(__double_as_longlong(x) + ((long long)k << 52));
}
__device__ __forceinline__ double qr_pow2(int k) { return __longlong_as_double((long long)(1023 + k) << 52); }
// a positive normal double of FP32's range to FP32 (cut off) and back, by the bits
__device__ __forceinline__ float qr_f32(double x) {
  const long long u = __double_as_longlong(x);
  return __uint_as_float((unsigned)((u >> 29) - (896ll << 23)));
}
__device__ __forceinline__ double qr_f64(float x) {
  return __longlong_as_double(((long long)__float_as_uint(x) << 29) + (896ll << 52));
}
// y = 1 / sqrt(v) and q = sqrt(v), v in [1, 8), from an FP32 seed y0 by the
// binomial series (1 - r)^-1/2 = 1 + r / 2 + 3 r^2 / 8 of r = 1 - v y0^2
__device__ __forceinline__ void qr_roots(double v, double& y, double& q) {
  const double y0 = qr_f64(rsqrtf(qr_f32(v)));
  const double t = v * y0, r = fma(-t, y0, 1.0), p = fma(0.375, r, 0.5);
  y = fma(y0 * r, p, y0);
  q = fma(t * r, p, t);
}
// 1 / v, v a normal number with a normal reciprocal: the geometric series
// 1 / (1 - r) = 1 + r + r^2 of r = 1 - m y0 on an FP32 seed y0
__device__ __forceinline__ double qr_rcp(double v) {
  const int e = qr_exp(v) - 1023;
  const double m = qr_scale(v, -e);  // [1, 2)
  const double y0 = qr_f64(1.f / qr_f32(m)), r = fma(-m, y0, 1.0);
  return qr_scale(fma(y0, fma(r, r, r), y0), -e);
}

// Reflector of column j from s = sum of |x|^2 over its rows from j on, by a
// whole warp: v_0 = x_0 - alpha into a[j], tau and (ALPHA) alpha.
template <bool ALPHA>
__device__ __forceinline__ void qr_reflect(cplx* a, int j, double s, int lane, double* tau, cplx* alph) {
  const cplx x0 = a[j];
  double t = 0.0;
  cplx al = cmk(0.0, 0.0), v0 = x0;
  // zero column, or one so small that tau would overflow (||x|| < 1e-150)
  if (!(s < INFINITY)) {
    al = cmk(-s, 0.0);
  } else if (s >= 1e-300) {
    // ||x|| and |x_0| by lanes of the same instructions: both scaled to [1, 8)
    const int e2 = (qr_exp(s) - 1023) & ~1;
    const int ex = max(qr_exp(x0.x), qr_exp(x0.y)) - 1023;
    const bool has = ex > -1023 + 60;
    const double ux = has ? qr_scale(x0.x, -ex) : 1.0, uy = has ? qr_scale(x0.y, -ex) : 0.0;
    const double a2 = fma(ux, ux, uy * uy);
    double y, q;
    qr_roots((lane & 1) ? a2 : qr_scale(s, -e2), y, q);
    const double ys = __shfl_xor_sync(0xffffffffu, y, 1), qs = __shfl_xor_sync(0xffffffffu, q, 1);
    const double nx = qr_scale((lane & 1) ? qs : q, e2 / 2);
    const double ya = (lane & 1) ? y : ys;
    const double ax0 = has ? qr_scale((lane & 1) ? q : qs, ex) : 0.0;
    // the phase of a leading entry negligible against ||x|| is not used
    const cplx ph = (ax0 > 1e-15 * nx) ? cmk(ux * ya, uy * ya) : cmk(1.0, 0.0);
    const double d = ax0 + nx;
    if (ALPHA) al = cscale(ph, -nx);
    v0 = cscale(ph, d);  // x_0 - alpha
    t = qr_rcp(nx * d);
  }
  __syncwarp();  // every lane has read x_0
  if (lane == 0) {
    a[j] = v0;
    *tau = t;
    if (ALPHA) *alph = al;
  }
}

// sum of |x|^2 over the rows from j on, by a whole warp
__device__ __forceinline__ double qr_norm2(const cplx* a, int j, int M, int lane) {
  double s = 0.0;
  for (int r = (j & ~31) + lane; r < M; r += 32)
    if (r >= j) s = fma(a[r].x, a[r].x, fma(a[r].y, a[r].y, s));
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  return s;
}

// a = column j + 1 <- H_j a with reflector v, then its reflector, by a whole warp
template <bool ALPHA>
__device__ __forceinline__ void qr_next(const cplx* v, cplx* a, int j, int M, const double t, int lane, double* tau,
                                        cplx* alph) {
  double s = 0.0;
  if (t != 0.0) {
    double re = 0.0, im = 0.0;
    for (int r = (j & ~31) + lane; r < M; r += 32) {
      if (r < j) continue;
      const cplx x = v[r], y = a[r];
      re = fma(x.x, y.x, fma(x.y, y.y, re));
      im = fma(x.x, y.y, fma(-x.y, y.x, im));
    }
    const cplx g = qr_csum<32>(re, im, lane, 0xffffffffu);
    const double sr = t * g.x, si = t * g.y;
    for (int r = (j & ~31) + lane; r < M; r += 32) {
      if (r < j) continue;
      const cplx x = v[r];
      cplx y = a[r];
      y.x = fma(-x.x, sr, fma(x.y, si, y.x));
      y.y = fma(-x.x, si, fma(-x.y, sr, y.y));
      a[r] = y;
      if (r > j) s = fma(y.x, y.x, fma(y.y, y.y, s));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  } else {
    s = qr_norm2(a, j + 1, M, lane);
  }
  __syncwarp();
  qr_reflect<ALPHA>(a, j + 1, s, lane, tau, alph);
}

// c <- H c, H = I - t v v^H, over the rows from j on, by a group of QR_G lanes
__device__ __forceinline__ void qr_apply(const cplx* v, cplx* c, int j, int M, double t, int gl, unsigned mask) {
  double re = 0.0, im = 0.0;
  for (int r = (j & ~(QR_G - 1)) + gl; r < M; r += QR_G) {
    if (r < j) continue;
    const cplx x = v[r], y = c[r];
    re = fma(x.x, y.x, fma(x.y, y.y, re));
    im = fma(x.x, y.y, fma(-x.y, y.x, im));
  }
  const cplx g = qr_csum<QR_G>(re, im, gl, mask);
  const double sr = t * g.x, si = t * g.y;
  for (int r = (j & ~(QR_G - 1)) + gl; r < M; r += QR_G) {
    if (r < j) continue;
    const cplx x = v[r];
    cplx y = c[r];
    y.x = fma(-x.x, sr, fma(x.y, si, y.x));
    y.y = fma(-x.x, si, fma(-x.y, sr, y.y));
    c[r] = y;
  }
}

// Column c of Q = H_0 ... H_{L-1} [I; 0], i.e. H_c, ..., H_0 applied to e_c
// (H_j leaves e_c alone for j > c), by a whole warp: the column in registers,
// row lane + 32 k in x[k], for M <= 32 R.  The reflectors that start in row
// block s are one loop whose blocks are known at compile time: blocks left out
// by a condition at run time would be predicated FP64 instructions, which take
// the pipe's time all the same (at eight blocks for 64 rows 1.5 ms for 256
// 64 x 42 matrices, against 0.6).
template <int R>
__device__ __forceinline__ void qr_qcol_r(const cplx* V, const double* tau, cplx* q, int c, int M, int lane) {
  cplx x[R];
#pragma unroll
  for (int k = 0; k < R; ++k) x[k] = cmk(lane + 32 * k == c ? 1.0 : 0.0, 0.0);
#pragma unroll
  for (int s = R - 1; s >= 0; --s) {
    for (int j = min(c, 32 * s + 31); j >= 32 * s; --j) {
      const double t = tau[j];
      if (t == 0.0) continue;
      const cplx* v = V + (int64_t)j * M;
      cplx y[R];
      double re = 0.0, im = 0.0;
#pragma unroll
      for (int k = s; k < R; ++k) {
        const int r = lane + 32 * k;
        y[k] = (r >= j && r < M) ? v[r] : cmk(0.0, 0.0);
        re = fma(y[k].x, x[k].x, fma(y[k].y, x[k].y, re));
        im = fma(y[k].x, x[k].y, fma(-y[k].y, x[k].x, im));
      }
      const cplx g = qr_csum<32>(re, im, lane, 0xffffffffu);
      const double sr = t * g.x, si = t * g.y;
#pragma unroll
      for (int k = s; k < R; ++k) {
        x[k].x = fma(-y[k].x, sr, fma(y[k].y, si, x[k].x));
        x[k].y = fma(-y[k].x, si, fma(-y[k].y, sr, x[k].y));
      }
    }
  }
#pragma unroll
  for (int k = 0; k < R; ++k)
    if (lane + 32 * k < M) q[lane + 32 * k] = x[k];
}

__device__ __forceinline__ void qr_qcol(const cplx* V, const double* tau, cplx* q, int c, int M, int lane) {
  switch ((M + 31) / 32) {
    case 1: return qr_qcol_r<1>(V, tau, q, c, M, lane);
    case 2: return qr_qcol_r<2>(V, tau, q, c, M, lane);
    case 3: return qr_qcol_r<3>(V, tau, q, c, M, lane);
    case 4: return qr_qcol_r<4>(V, tau, q, c, M, lane);
    default: break;
  }
  for (int r = lane; r < M; r += 32) q[r] = cmk(r == c ? 1.0 : 0.0, 0.0);
  for (int j = c; j >= 0; --j) {
    const double t = tau[j];
    if (t == 0.0) continue;
    const cplx* v = V + (int64_t)j * M;
    double re = 0.0, im = 0.0;
    for (int r = (j & ~31) + lane; r < M; r += 32) {
      if (r < j) continue;
      const cplx y = v[r], x = q[r];
      re = fma(y.x, x.x, fma(y.y, x.y, re));
      im = fma(y.x, x.y, fma(-y.y, x.x, im));
    }
    const cplx g = qr_csum<32>(re, im, lane, 0xffffffffu);
    const double sr = t * g.x, si = t * g.y;
    for (int r = (j & ~31) + lane; r < M; r += 32) {
      if (r < j) continue;
      const cplx y = v[r];
      cplx x = q[r];
      x.x = fma(-y.x, sr, fma(y.y, si, x.x));
      x.y = fma(-y.x, si, fma(-y.y, sr, x.y));
      q[r] = x;
    }
  }
}

// Order in which warp w >= 1 of a CTA takes the columns right of the next one:
// two rounds over the quarters without warp 0, then all quarters in turn (the
// chain is worth one to two of a quarter's tasks).
__device__ __forceinline__ int qr_slot(int w) {
  const int s = w & 3, q = w >> 2;
  if (s == 0) return 6 + (q - 1) * 4;
  return q < 2 ? q * 3 + s - 1 : 6 + (q - 2) * 4 + s;
}

// QR with explicit Q of one problem (stage QS) by the whole CTA (a multiple of
// 128 threads); tau / alph >= l entries of shared memory.
template <int QS>
__device__ __forceinline__ void qr_dev(const Dims& D, const ProbPtr& P, double* tau, cplx* alph) {
  const int M = (QS == QR_Y) ? D.m : D.n;
  const int L = D.l;
  cplx* A = (QS == QR_Y) ? P.Y : P.Yt;
  cplx* Qo = (QS == QR_Y) ? P.Q : P.Qt;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = blockDim.x >> 5;
  const int gl = lane & (QR_G - 1), half = lane / QR_G;
  const unsigned gmask = ((1u << QR_G) - 1u) << (lane & ~(QR_G - 1));
  const int slot = qr_slot(warp);
  if (warp == 0) qr_reflect<QS == QR_BH>(A, 0, qr_norm2(A, 0, M, lane), lane, tau, alph);
  __syncthreads();
  for (int j = 0; j + 1 < L; ++j) {
    const double t = tau[j];
    const cplx* v = A + (int64_t)j * M;
    if (warp == 0)
      qr_next<QS == QR_BH>(v, A + (int64_t)(j + 1) * M, j, M, t, lane, tau + j + 1, alph + j + 1);
    else if (t != 0.0)
      for (int c = j + 2 + 2 * slot + half; c < L; c += 2 * (nw - 1)) qr_apply(v, A + (int64_t)c * M, j, M, t, gl, gmask);
    __syncthreads();
  }
  // X = Rb^H (lower triangle, column-major L x L) for the SVD of B: element
  // (r, c) of X is conj(Rb[c][r]), Rb[i][c] = A[c M + i] above the diagonal
  // and alpha_c on it
  if (QS == QR_BH) {
    for (int e = tid; e < L * L; e += blockDim.x) {
      const int c = e / L, r = e % L;
      cplx v = cmk(0.0, 0.0);
      if (c < r) v = cconj(A[(int64_t)r * M + c]);
      else if (c == r) v = cconj(alph[c]);
      P.R[(int64_t)c * L + r] = v;
    }
  }
  for (int c = L - 1 - warp; c >= 0; c -= nw) qr_qcol(A, tau, Qo + (int64_t)c * M, c, M, lane);
  __syncthreads();
}

enum { JAC_MAXSWEEPS = 60, JAC_G = 8 };

// x_a' = c u - conj(se) v, x_b' = se u + c v, each part three operations in a
// fixed order (every Jacobi kernel gives the same bits)
__device__ __forceinline__ void jac_rotate(double c, cplx se, cplx u, cplx v, cplx& xa, cplx& xb) {
  xa = cmk(fma(-se.y, v.y, fma(-se.x, v.x, __dmul_rn(c, u.x))), fma(se.y, v.x, fma(-se.x, v.y, __dmul_rn(c, u.y))));
  xb = cmk(fma(-se.y, u.y, fma(se.x, u.x, __dmul_rn(c, v.x))), fma(se.y, u.x, fma(se.x, u.y, __dmul_rn(c, v.y))));
}

// One lane's part of x_a^H x_b
struct JacDot {
  double re = 0.0, im = 0.0;
  __device__ __forceinline__ void add(cplx u, cplx v) {
    re = fma(u.x, v.x, fma(u.y, v.y, re));
    im = fma(u.x, v.y, fma(-u.y, v.x, im));
  }
};
// x_a^H x_b from the four parts each of the JAC_G lanes of a group holds
__device__ __forceinline__ cplx jac_gram(const JacDot* d, int lane, unsigned mask) {
  return qr_csum<8>((d[0].re + d[2].re) + (d[1].re + d[3].re), (d[0].im + d[2].im) + (d[1].im + d[3].im), lane, mask);
}
// the same from the one part of each lane of a warp (part m in lanes 8 m .. 8 m + 7)
__device__ __forceinline__ cplx jac_gram_warp(JacDot d, int lane) {
#pragma unroll
  for (int o = 16; o >= 8; o >>= 1) {
    d.re += __shfl_xor_sync(0xffffffffu, d.re, o);
    d.im += __shfl_xor_sync(0xffffffffu, d.im, o);
  }
  return qr_csum<8>(d.re, d.im, lane, 0xffffffffu);
}

__device__ __forceinline__ void jacobi_finish(const Dims& D, const ProbPtr& P, double* sv, int* perm);

// Rotation of a pair: x_a' = c x_a - conj(se) x_b, x_b' = se x_a + c x_b that
// makes them orthogonal, from aa = |x_a|^2, bb = |x_b|^2, g = x_a^H x_b and
// ag2 = |g|^2; tg = t |g|, what the squared norms change by.  About 30 FP64
// operations: |g| and 1 / |g| from one Newton reciprocal root, the tangent t
// from FP32 and one Newton step of t^2 + 2 zeta t - 1 = 0 (relative error
// ~1e-14; c and s = c t are unitary to FP64 whatever t is).  Eight lanes
// repeat them, so the ~140 operations of the library's roots and divisions
// were as much FP64 work as the rows of a 40-row pair.
__device__ __forceinline__ void jac_rotation(double aa, double bb, cplx g, double ag2, double& c, cplx& se, double& tg) {
  // |g|^2 = w 2^e2, w in [1, 4)
  const int e2 = (qr_exp(ag2) - 1023) & ~1;
  const double w = ag2 * qr_pow2(-e2);
  double y, q;
  qr_roots(w, y, q);
  const double inv = y * qr_pow2(-(e2 / 2)), ag = q * qr_pow2(e2 / 2);
  const cplx e = cscale(g, inv);
  const double zeta = (0.5 * (bb - aa)) * inv;
  const float zf = fabsf((float)zeta);
  const float tf = zf > 1e9f ? 0.5f / zf : 1.f / (zf + sqrtf(fmaf(zf, zf, 1.f)));
  const double t0 = (double)tf, az = fabs(zeta);
  const double res = fma(t0, t0 + 2.0 * az, -1.0);
  const double t1 = t0 - (double)((float)res / (2.f * (tf + zf)));
  const double t = zeta >= 0.0 ? t1 : -t1;
  qr_roots(fma(t, t, 1.0), c, q);
  se = cscale(e, c * t);
  tg = __dmul_rn(t, ag);  // (a product of its own: the callers' sums must not contract with it)
}

// One-sided Jacobi SVD of one problem by the whole CTA (any multiple of
// JAC_G threads, at least 32); sv, nrm, perm >= l entries and red >= 32
// doubles of shared memory, rotated one shared int.
__device__ __forceinline__ void jacobi_dev(const Dims& D, const ProbPtr& P, int* status, double* sv, double* nrm,
                                           int* perm, int* rotated_p, double* red) {
  int& rotated = *rotated_p;
  const int L = D.l;
  cplx* X = P.R;
  cplx* J = P.J;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = blockDim.x >> 5;
  const int gl = lane & (JAC_G - 1);                      // lane within its group
  const int grp = tid / JAC_G, ngrp = blockDim.x / JAC_G;  // group index, groups per CTA
  const unsigned gmask = ((1u << JAC_G) - 1u) << (lane & ~(JAC_G - 1));
  double f2 = 0.0;
  if (D.js == 0)
    for (int e = tid; e < L * L; e += blockDim.x) J[e] = cmk((e / L) == (e % L) ? 1.0 : 0.0, 0.0);
  if (tid < RED_LANES)
    for (int e = tid; e < L * L; e += RED_LANES) f2 += cabs2(X[e]);
  f2 = block_sum(f2, red);
  const int Lp = (L + 1) & ~1;
  const double eps = 2.220446049250313e-16;
  const double tol = 4.0 * eps * sqrt((double)L);
  const double small = ((double)L * eps) * ((double)L * eps) * f2;
  int sweep = D.js == 2 ? JAC_MAXSWEEPS + 1 : 0;
  for (; sweep < JAC_MAXSWEEPS; ++sweep) {
    // exact squared column norms at the start of every sweep; within the sweep
    // they follow each rotation: |x_a'|^2 = |x_a|^2 - t|g|, |x_b'|^2 = |x_b|^2 + t|g|
    for (int c = warp; c < L; c += nw) {
      const cplx* xc = X + (int64_t)c * L;
      double s2 = 0.0;
      for (int r = lane; r < L; r += 32) s2 += cabs2(xc[r]);
      s2 = warp_sum(s2);
      if (lane == 0) nrm[c] = s2;
    }
    if (tid == 0) rotated = 0;
    __syncthreads();
    for (int rnd = 0; rnd < Lp - 1; ++rnd) {
      for (int pi = grp; pi < Lp / 2; pi += ngrp) {
        int a, b;
        if (pi == 0) { a = Lp - 1; b = rnd; }
        else { a = (rnd + pi) % (Lp - 1); b = (rnd - pi + (Lp - 1)) % (Lp - 1); }
        if (a > b) { const int t = a; a = b; b = t; }
        if (b >= L) continue;  // uniform over the group
        cplx* xa = X + (int64_t)a * L;
        cplx* xb = X + (int64_t)b * L;
        const double aa = nrm[a], bb = nrm[b];
        if (aa <= small || bb <= small) continue;
        JacDot dot[4];  // rows gl + 8 m + 32 k in dot[m], as the lanes of k_jacobi_cl's warps take them
        int r = gl;
        for (; r + 24 < L; r += 32) {
#pragma unroll
          for (int m = 0; m < 4; ++m) dot[m].add(xa[r + 8 * m], xb[r + 8 * m]);
        }
        if (r < L) dot[0].add(xa[r], xb[r]);
        if (r + 8 < L) dot[1].add(xa[r + 8], xb[r + 8]);
        if (r + 16 < L) dot[2].add(xa[r + 16], xb[r + 16]);
        const cplx g = jac_gram(dot, lane, gmask);
        const double ag2 = fma(g.x, g.x, __dmul_rn(g.y, g.y));
        if (!(ag2 > tol * tol * (aa * bb)) || ag2 < 2.2250738585072014e-308) continue;  // (below normal numbers)
        double c, tg;
        cplx se;
        jac_rotation(aa, bb, g, ag2, c, se, tg);
        for (r = gl; r < L; r += JAC_G) jac_rotate(c, se, xa[r], xb[r], xa[r], xb[r]);
        cplx* ja = J + (int64_t)a * L;
        cplx* jb = J + (int64_t)b * L;
        for (r = gl; r < L; r += JAC_G) jac_rotate(c, se, ja[r], jb[r], ja[r], jb[r]);
        if (gl == 0) {
          nrm[a] = aa - tg;
          nrm[b] = bb + tg;
          rotated = 1;
        }
      }
      __syncthreads();
    }
    const int any = rotated;
    __syncthreads();
    if (!any) break;
  }
  if (sweep == JAC_MAXSWEEPS && tid == 0) atomicOr(status, 2);  // not converged (non-fatal)
  jacobi_finish(D, P, sv, perm);
}

// After the sweeps (X = P.R holds X J = W S, J = P.J): singular values =
// column norms, sorted descending (ties by lower index; a NaN value ranks
// below every number, so perm is a permutation of 0..L-1 whatever the input),
// Jk = the leading k normalised columns of X J, Wk = the matching columns of J.
__device__ __forceinline__ void jacobi_finish(const Dims& D, const ProbPtr& P, double* sv, int* perm) {
  const int L = D.l, K = D.k;
  const cplx* X = P.R;
  const cplx* J = P.J;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = blockDim.x >> 5;
  for (int c = warp; c < L; c += nw) {
    const cplx* xc = X + (int64_t)c * L;
    double s = 0.0;
    for (int r = lane; r < L; r += 32) s += cabs2(xc[r]);
    s = warp_sum(s);
    if (lane == 0) sv[c] = sqrt(s);
  }
  __syncthreads();
  for (int c = tid; c < L; c += blockDim.x) {
    const double s = (sv[c] == sv[c]) ? sv[c] : -1.0;
    int rk = 0;
    for (int j = 0; j < L; ++j) {
      const double t = (sv[j] == sv[j]) ? sv[j] : -1.0;
      rk += (t > s) || (t == s && j < c);
    }
    perm[rk] = c;
  }
  __syncthreads();
  for (int i = tid; i < L; i += blockDim.x) P.sigma[i] = sv[perm[i]];
  for (int e = tid; e < K * L; e += blockDim.x) {
    const int t = e / L, r = e % L;
    const int c = perm[t];
    const double s = sv[c];
    P.Jk[e] = (s > 0.0) ? cscale(X[(int64_t)c * L + r], 1.0 / s) : cmk(0.0, 0.0);
    P.Wk[e] = J[(int64_t)c * L + r];
  }
}

// ---------------------------------------------------------------------------
// TEBD stages: the size plan of a bond, theta~ (contraction and gate), and
// the rebuild after truncation (tebd_kernels.cu documents each).
// ---------------------------------------------------------------------------
// Sizes of one bond from its current bond dimensions (see k_plan).
__device__ __forceinline__ Dims plan_dev(const ProbPtr& P, int p, int digits) {
  Dims D;
  D.dl = P.dl_s;
  D.dr = P.dr_s;
  D.cl = *P.chi_l;
  D.cm = *P.chi_m;
  D.cr = *P.chi_r;
  D.m = D.dl * D.cl;
  D.n = D.dr * D.cr;
  const int k = min(P.chicap, min(D.m, D.n));
  D.k = k;
  D.l = min(k + p, min(D.m, D.n));
  D.bond = P.bond_s;
  D.chain = P.chain_s;
  D.active = (D.cm > 0) ? 1 : 0;
  D.r = 0;
  D.chk = 0;
  D.qflag = 0;
  D.dig = (digits && dp_rule(D.m, D.n, D.l)) ? 1 : 0;
  D.cq = 0;
  D.cf = 0;
  D.js = 0;
  D.gr = 0;
  return D;
}

enum { TH_TK = 16, TH_MAXR = 64 };

// One (alpha, beta) block (ablk, bblk) of theta~ by a CTA of 256 threads
// (see k_theta); th_sm holds 2 TH_TK TH_MAXR + TH_MAXR^2 complex numbers.
__device__ __forceinline__ void theta_tile_dev(const Dims& D, const ProbPtr& P, int ablk, int bblk,
                                               int identity_gate, cplx* th_sm) {
  const int dl = D.dl, dr = D.dr, cl = D.cl, cm = D.cm, cr = D.cr;
  const int TA = max(1, 32 / dl), TB = max(1, 32 / dr);
  const int a0 = ablk * TA, b0 = bblk * TB;
  if (a0 >= cl || b0 >= cr) return;
  const int ta = min(TA, cl - a0), tb = min(TB, cr - b0);
  const int rows = dl * ta, cols = dr * tb;  // <= 64 each
  cplx* Ls = th_sm;                          // [TH_TK][TH_MAXR]
  cplx* Rs = Ls + TH_TK * TH_MAXR;           // [TH_TK][TH_MAXR]
  cplx* Cs = Rs + TH_TK * TH_MAXR;           // [rows][cols]
  const int tid = threadIdx.x;
  const int nout = rows * cols;
  cplx acc[16];
#pragma unroll
  for (int s = 0; s < 16; ++s) acc[s] = cmk(0.0, 0.0);
  const cplx* gl = P.gl;
  const cplx* gr = P.gr;
  for (int g0 = 0; g0 < cm; g0 += TH_TK) {
    // L rows (i', a): lam_l[a] Gl[i'][a0+a][g] lam_m[g]; g fastest
    for (int e = tid; e < TH_TK * rows; e += 256) {
      const int kk = e % TH_TK, ri = e / TH_TK;
      const int ip = ri / ta, a = ri % ta, g = g0 + kk;
      cplx v = cmk(0.0, 0.0);
      if (g < cm) {
        v = gl[((int64_t)ip * P.cap_l + a0 + a) * P.cap_m + g];
        v = cscale(v, P.laml[a0 + a] * P.lamm[g]);
      }
      Ls[kk * TH_MAXR + ri] = v;
    }
    // R columns (j', c): Gr[j'][g][b0+c] lam_r[c]; c fastest
    for (int e = tid; e < TH_TK * cols; e += 256) {
      const int c = e % tb, rest = e / tb;
      const int jp = rest % dr, kk = rest / dr;
      const int g = g0 + kk;
      cplx v = cmk(0.0, 0.0);
      if (g < cm) {
        v = gr[((int64_t)jp * P.cap_m + g) * P.cap_r + b0 + c];
        v = cscale(v, P.lamr[b0 + c]);
      }
      Rs[kk * TH_MAXR + jp * tb + c] = v;
    }
    __syncthreads();
#pragma unroll
    for (int s = 0; s < 16; ++s) {
      const int o = tid + 256 * s;
      if (o < nout) {
        const int ri = o / cols, ci = o % cols;
        cplx a = acc[s];
#pragma unroll 4
        for (int kk = 0; kk < TH_TK; ++kk) cfma(a, Ls[kk * TH_MAXR + ri], Rs[kk * TH_MAXR + ci]);
        acc[s] = a;
      }
    }
    __syncthreads();
  }
#pragma unroll
  for (int s = 0; s < 16; ++s) {
    const int o = tid + 256 * s;
    if (o < nout) Cs[o] = acc[s];
  }
  __syncthreads();
  // gate: rows of Cs are (i', a) = i'*ta + a, columns (j', c) = j'*tb + c.
  // A bond whose gate is applied as a GEMM gets its pre-gate theta in Cpre.
  const int dd = dl * dr;
  const bool pre = !identity_gate && P.Cpre != nullptr;
  cplx* th = pre ? P.Cpre : const_cast<cplx*>(P.theta);
  for (int o = tid; o < nout; o += 256) {
    const int ri = o / cols, ci = o % cols;
    const int i = ri / ta, a = ri % ta, j = ci / tb, c = ci % tb;
    const cplx* grow = P.gate + (int64_t)(i * dr + j) * dd;
    cplx v = cmk(0.0, 0.0);
    if (identity_gate || pre)
      v = Cs[(i * ta + a) * cols + j * tb + c];
    else
      for (int ip = 0; ip < dl; ++ip)
        for (int jp = 0; jp < dr; ++jp) cfma(v, grow[ip * dr + jp], Cs[(ip * ta + a) * cols + jp * tb + c]);
    th[(int64_t)(i * cl + a0 + a) * D.n + j * cr + b0 + c] = v;
  }
}

// Truncation, renormalisation and Gamma rebuild of one bond by the whole CTA
// (see k_rebuild), or by `parts` CTAs of which this is `part`: each finds the
// rank itself and the first one writes what there is once per bond.
// s_rank_p / s_inv_p point at shared scratch.
__device__ __forceinline__ void rebuild_dev(const Dims& D, const ProbPtr& P, double cutoff, double* wout_p,
                                            int* status, int* s_rank_p, double* s_inv_p, int part = 0,
                                            int parts = 1) {
  if (threadIdx.x == 0) {
    double nf = 0.0;
    for (int i = 0; i < NPART; ++i) nf += P.part[i];
    const double s0 = P.sigma[0];
    int r = 0;
    double kept = 0.0;
    const bool finite = isfinite(nf) && isfinite(s0);
    if (finite && s0 > 0.0) {
      while (r < D.k && P.sigma[r] > cutoff * s0) {
        kept += P.sigma[r] * P.sigma[r];
        ++r;
      }
    }
    if (!finite || r == 0 || !isfinite(kept)) {
      if (part == 0) atomicOr(status, 1);
      r = 0;
    }
    (*s_rank_p) = r;
    (*s_inv_p) = (r > 0) ? 1.0 / sqrt(kept) : 0.0;
    if (part == 0) *wout_p = (r > 0 && nf > 0.0) ? 1.0 - kept / nf : 0.0;
  }
  __syncthreads();
  const int r = (*s_rank_p);
  if (r == 0) return;
  double* lam = const_cast<double*>(P.lamm);
  const int capm = P.cap_m;
  if (part == 0)
    for (int i = threadIdx.x; i < capm; i += blockDim.x) lam[i] = (i < r) ? P.sigma[i] * (*s_inv_p) : 0.0;
  const int64_t e0 = (int64_t)part * blockDim.x + threadIdx.x, es = (int64_t)parts * blockDim.x;
  cplx* gl = const_cast<cplx*>(P.gl);
  cplx* gr = const_cast<cplx*>(P.gr);
  const int dl = D.dl, dr = D.dr, cl = D.cl, cr = D.cr, K = D.k;
  for (int64_t e = e0; e < (int64_t)dl * cl * r; e += es) {
    const int g = (int)(e % r);
    const int row = (int)(e / r);  // i*cl + a
    const int a = row % cl, i = row / cl;
    const double ll = P.laml[a];
    const cplx u = P.U[(int64_t)row * K + g];
    gl[((int64_t)i * P.cap_l + a) * capm + g] = (ll > 0.0) ? cscale(u, 1.0 / ll) : cmk(0.0, 0.0);
  }
  for (int64_t e = e0; e < (int64_t)dr * r * cr; e += es) {
    const int c = (int)(e % cr);
    const int rest = (int)(e / cr);
    const int g = rest % r, j = rest / r;
    const double lr = P.lamr[c];
    const cplx v = P.V[(int64_t)g * D.n + j * cr + c];
    gr[((int64_t)j * capm + g) * P.cap_r + c] = (lr > 0.0) ? cscale(v, 1.0 / lr) : cmk(0.0, 0.0);
  }
  __syncthreads();
  if (part == 0 && threadIdx.x == 0) *P.chi_m = r;
}

}  // namespace tg
