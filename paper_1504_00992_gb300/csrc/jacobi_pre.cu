// Small SVD by an FP32 Jacobi and digit-split corrections (sm_103a): X J = W S
// for X = Rb^H (Section IV's step ii) to FP64, for the problems whose other
// products run from digit splits.
//
// The one-sided Jacobi kernels spend 14 l^3 FP64 (or double-float) multiply-
// adds per sweep and five to seven sweeps, nearly all of them far from the
// final accuracy.  Here
//   1. k_jac_pre runs the same sweeps in FP32 on X rounded to FP32 (columns
//      orthogonal to ~3e-6) and keeps the accumulated J;
//   2. J is made unitary to FP64 (J^H J from digits, k_lowdin64) and X J is
//      formed from digits;
//   3. up to JP_STEPS times, the first-order rotations of every pair at once:
//      with G = X^H X from digits, K_ab = t e from the pair's 2 x 2 problem
//      (Jacobi's angle t and phase e), X <- X T and J <- J T with
//      T = I + K + K^2 / 2, K skew-Hermitian, so that T is unitary to K^4 / 4.
//      The residual falls from ~3e-6 to its square over the gap (and 1e-7 of
//      it, K is FP32), i.e. below FP64's tolerance in two steps;
//   4. a problem whose columns are orthogonal to the Jacobi kernels' own
//      tolerance is done; the others go on in those kernels from (X, J).
// Pairs with an angle above JP_ANGLE (nearly equal singular values) are left
// out of K and so to step 4, where each costs one rotation.
//
// Graded columns (TEBD spectra reach 1e-14): the products X J and X T scale
// the left operand's columns by S = 2^-e of their norms and the right one's
// rows by S^-1, so that every column of the result is rounded relative to its
// own norm and not to the largest singular value.
//
// Measured, l = 120: 16 problems in FP64 14.1 ms in the cluster Jacobi alone,
// 4.9 ms here (FP32 sweeps 2.7, products 0.4, corrections 0.7, the Jacobi
// kernel's check and ranking 1.1); 152 in double-float 10.3 ms, against 6.1.
// The sweeps are bound by the latency of a round (a barrier, two trips to
// shared memory, two to J in L1).
//
// FP32 kernel: X in shared memory for l <= JP_MAXL (205 KB), J through L1/L2,
// one group of eight lanes per pair, the pair's columns in registers between
// the inner product and the rotation.
#include <cooperative_groups.h>
#include <cuda_runtime.h>
#include <math.h>

#include "dfsplit.cuh"
#include "internal.cuh"
#include "mixed.cuh"
#include "once.cuh"
#include "profiler.cuh"
#include "stages.cuh"

namespace cg = cooperative_groups;

namespace tg {

enum { JP_MAXL = 160, JP_G = 8, JP_ROWS = JP_MAXL / JP_G, JP_THREADS = 640, JP_SWEEPS = 12, JP_STEPS = 2 };
static const float JP_TOL = 3e-6f;    // cosine of a pair the FP32 sweeps leave alone
static const float JP_ANGLE = 3e-5f;  // largest angle of a first-order rotation

__device__ __forceinline__ bool jp_takes(const Dims& D, int cond) {
  return D.active && !((cond & DPC_DIG) && !D.dig) && !((cond & DPC_WIDE) && D.l < DP_WIDE_L);
}

__device__ __forceinline__ float2 jp_shfl_sum(float2 v, unsigned mask) {
#pragma unroll
  for (int o = JP_G / 2; o > 0; o >>= 1) {
    v.x += __shfl_xor_sync(mask, v.x, o);
    v.y += __shfl_xor_sync(mask, v.y, o);
  }
  return v;
}

// x 2^k by the exponent bits, to FP32 (0 below its range)
__device__ __forceinline__ float jp_f32(double x, int k) {
  const long long u = __double_as_longlong(x);
  const int e = (int)((u >> 52) & 0x7FF) + k;
  return (((u >> 52) & 0x7FF) == 0 || e <= 1023 - 126) ? 0.f : (float)__longlong_as_double(u + ((long long)k << 52));
}
__device__ __forceinline__ int jp_exp2(double x) { return (int)((__double_as_longlong(x) >> 52) & 0x7FF) - 1023; }

// Rotation of a pair from its squared norms and g = x_a^H x_b; false where the
// cosine is below JP_TOL.  tg: what the squared norms change by.
struct JpRot {
  float c, sx, sy, tg;
};
__device__ __forceinline__ bool jp_rotation(float na, float nb, float gx, float gy, JpRot& R) {
  const float ra = rsqrtf(na), rb = rsqrtf(nb);
  const float cx = (gx * ra) * rb, cy = (gy * ra) * rb;  // the cosine
  const float co = sqrtf(fmaf(cx, cx, cy * cy));
  if (!(co > JP_TOL)) return false;
  const float ic = 1.f / co, ex = cx * ic, ey = cy * ic;
  // zeta = (nb - na) / (2 |g|) with |g| = co sqrt(na nb)
  const float zeta = ((nb - na) * ra) * rb * (0.5f * ic);
  const float az = fabsf(zeta);
  const float t = (zeta >= 0.f ? 1.f : -1.f) / (az > 1e9f ? 2.f * az : az + sqrtf(fmaf(zeta, zeta, 1.f)));
  const float s = rsqrtf(fmaf(t, t, 1.f));
  R.c = s;
  R.sx = s * t * ex;
  R.sy = s * t * ey;
  R.tg = t * (co / (ra * rb));
  return true;
}
__device__ __forceinline__ void jp_rotate(const JpRot& R, float2 u, float2 v, float2& xa, float2& xb) {
  xa = make_float2(fmaf(R.c, u.x, -fmaf(R.sx, v.x, R.sy * v.y)), fmaf(R.c, u.y, -fmaf(R.sx, v.y, -R.sy * v.x)));
  xb = make_float2(fmaf(R.c, v.x, fmaf(R.sx, u.x, -R.sy * u.y)), fmaf(R.c, v.y, fmaf(R.sx, u.y, R.sy * u.x)));
}

__global__ void __launch_bounds__(JP_THREADS) k_jac_pre(Dims* dims, const ProbPtr* __restrict__ ptrs, int cond) {
  extern __shared__ __align__(16) unsigned char jp_raw[];
  __shared__ float nrm[JP_MAXL];
  __shared__ int s_exp;
  __shared__ int rotated;
  const int p = blockIdx.x;
  const Dims D = dims[p];
  if (!jp_takes(D, cond)) {
    if ((cond & DPC_WIDE) && threadIdx.x == 0) dims[p].js = 0;
    return;
  }
  const ProbPtr P = ptrs[p];
  const int L = D.l, tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, warp = tid >> 5, nw = nt >> 5;
  float2* X = reinterpret_cast<float2*>(jp_raw);
  // FP32 J in the upper half of the buffer its FP64 form fills at the end
  float2* J = reinterpret_cast<float2*>(P.J) + (size_t)L * L;
  if (tid == 0) s_exp = 0;
  __syncthreads();
  int e = 0;
  bool bad = false;
  for (int i = tid; i < L * L; i += nt) {
    const cplx v = P.R[i];
    e = max(e, max(oz_exp(v.x), oz_exp(v.y)));
    bad |= !isfinite(v.x) || !isfinite(v.y);
  }
  atomicMax(&s_exp, e);
  const bool any_bad = __syncthreads_or(bad);
  const int E = s_exp;
  if (any_bad || E == 0) {  // left to the Jacobi kernels as it is
    if (tid == 0) dims[p].js = 0;
    return;
  }
  const int up = 1023 - E;  // to max |x| in [1, 2)
  for (int i = tid; i < L * L; i += nt) {
    const cplx v = P.R[i];
    X[i] = make_float2(jp_f32(v.x, up), jp_f32(v.y, up));
    J[i] = make_float2((i / L) == (i % L) ? 1.f : 0.f, 0.f);
  }
  __syncthreads();
  const int gl = lane & (JP_G - 1), grp = tid / JP_G, ngrp = nt / JP_G;
  const unsigned gmask = ((1u << JP_G) - 1u) << (lane & ~(JP_G - 1));
  const int Lp = (L + 1) & ~1;
  for (int sweep = 0; sweep < JP_SWEEPS; ++sweep) {
    for (int c = warp; c < L; c += nw) {
      float s = 0.f;
      for (int r = lane; r < L; r += 32) {
        const float2 v = X[c * L + r];
        s = fmaf(v.x, v.x, fmaf(v.y, v.y, s));
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
      if (lane == 0) nrm[c] = s;
    }
    if (tid == 0) rotated = 0;
    __syncthreads();
    for (int rnd = 0; rnd < Lp - 1; ++rnd) {
      for (int pi = grp; pi < Lp / 2; pi += ngrp) {
        int a = pi == 0 ? Lp - 1 : rnd + pi, b = pi == 0 ? rnd : rnd - pi;
        if (pi > 0) {
          if (a >= Lp - 1) a -= Lp - 1;
          if (b < 0) b += Lp - 1;
        }
        if (a > b) {
          const int t = a;
          a = b;
          b = t;
        }
        if (b >= L) continue;  // uniform over the group
        const float na = nrm[a], nb = nrm[b];
        if (!(na > 1e-34f) || !(nb > 1e-34f)) continue;  // below FP32's squares
        float2* xa = X + a * L;
        float2* xb = X + b * L;
        float2 u[JP_ROWS], v[JP_ROWS];
        float2 g = make_float2(0.f, 0.f);
#pragma unroll
        for (int q = 0; q < JP_ROWS; ++q) {
          if (q * JP_G >= L) continue;  // uniform
          const int r = gl + q * JP_G;
          u[q] = r < L ? xa[r] : make_float2(0.f, 0.f);
          v[q] = r < L ? xb[r] : make_float2(0.f, 0.f);
          g.x = fmaf(u[q].x, v[q].x, fmaf(u[q].y, v[q].y, g.x));
          g.y = fmaf(u[q].x, v[q].y, fmaf(-u[q].y, v[q].x, g.y));
        }
        g = jp_shfl_sum(g, gmask);
        JpRot R;
        if (!jp_rotation(na, nb, g.x, g.y, R)) continue;
#pragma unroll
        for (int q = 0; q < JP_ROWS; ++q) {
          const int r = gl + q * JP_G;
          if (r < L) jp_rotate(R, u[q], v[q], xa[r], xb[r]);
        }
        float2* ja = J + (size_t)a * L;
        float2* jb = J + (size_t)b * L;
#pragma unroll
        for (int q = 0; q < JP_ROWS; ++q) {
          if (q * JP_G >= L) continue;
          const int r = gl + q * JP_G;
          u[q] = r < L ? ja[r] : make_float2(0.f, 0.f);
          v[q] = r < L ? jb[r] : make_float2(0.f, 0.f);
        }
#pragma unroll
        for (int q = 0; q < JP_ROWS; ++q) {
          const int r = gl + q * JP_G;
          if (r < L) jp_rotate(R, u[q], v[q], ja[r], jb[r]);
        }
        if (gl == 0) {
          nrm[a] = fmaxf(na - R.tg, 0.f);
          nrm[b] = nb + R.tg;
          rotated = 1;
        }
      }
      __syncthreads();
    }
    const int any = rotated;
    __syncthreads();
    if (!any) break;
  }
  // J to FP64 in place: in ascending order an entry's FP64 form overwrites
  // only FP32 entries already read
  for (int i0 = 0; i0 < L * L; i0 += nt) {
    const int i = i0 + tid;
    const float2 v = i < L * L ? J[i] : make_float2(0.f, 0.f);
    __syncthreads();
    if (i < L * L) P.J[i] = cmk((double)v.x, (double)v.y);
    __syncthreads();
  }
  // S from the columns of X itself
  for (int c = warp; c < L; c += nw) {
    int m = 0;
    for (int r = lane; r < L; r += 32) {
      const cplx v = P.R[(size_t)c * L + r];
      m = max(m, max(oz_exp(v.x), oz_exp(v.y)));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
    if (lane == 0) P.sigma[c] = m > 0 ? __longlong_as_double((long long)max(1, 2046 - m) << 52) : 1.0;
  }
  if (tid == 0) dims[p].js = 1;
}

// Squared norms (the diagonal of G), the exponents of S_c = 2^s_k[c] that
// bring them to [1, 4), and the square below which a column is negligible; by
// the whole CTA, with a barrier at the end.
__device__ __forceinline__ void jp_scales(const cplx* G, int L, float small_u, double* s_n, int* s_k, double* s_f2) {
  for (int c = threadIdx.x; c < L; c += blockDim.x) {
    const double n = G[(size_t)c * L + c].x;
    s_n[c] = n;
    s_k[c] = n > 0.0 ? -((jp_exp2(n) - ((jp_exp2(n) & 1) ? 1 : 0)) / 2) : 0;  // -floor(log2 n / 2)
  }
  __syncthreads();
  if (threadIdx.x < 32) {
    double f2 = 0.0;
    for (int c = threadIdx.x; c < L; c += 32) f2 += s_n[c];
    f2 = warp_sum(f2);
    if (threadIdx.x == 0) *s_f2 = (double)small_u * small_u * (double)L * (double)L * f2;
  }
  __syncthreads();
}

// K_ab = t e of a pair from g = x_a^H x_b, 0 where the angle is above JP_ANGLE
// or a column is negligible; worst: the largest cosine so far.
__device__ __forceinline__ float2 jp_angle(cplx g, double na, double nb, int ka, int kb, double small, float& worst) {
  if (!(na > small && nb > small)) return make_float2(0.f, 0.f);
  const float gx = jp_f32(g.x, ka + kb), gy = jp_f32(g.y, ka + kb);
  const float va = jp_f32(na, 2 * ka), vb = jp_f32(nb, 2 * kb);  // in [1, 4)
  const float ag = sqrtf(fmaf(gx, gx, gy * gy));
  const float co = ag * rsqrtf(va) * rsqrtf(vb);
  worst = (co > worst || co != co) ? co : worst;
  if (!(ag > 0.f)) return make_float2(0.f, 0.f);
  // zeta = (nb - na) / (2 |g|), scaled by S_a S_b above and below
  const double d = nb - na;
  const int ke = ka + kb;
  const float dz = jp_exp2(d) + ke > 120 ? (d > 0.0 ? 1e36f : -1e36f) : jp_f32(d, ke);
  const float zeta = dz / (2.f * ag), az = fabsf(zeta);
  const float t = (zeta >= 0.f ? 1.f : -1.f) / (az > 1e9f ? 2.f * az : az + sqrtf(fmaf(zeta, zeta, 1.f)));
  if (!(fabsf(t) <= JP_ANGLE)) return make_float2(0.f, 0.f);
  const float ia = 1.f / ag;
  return make_float2(t * (gx * ia), t * (gy * ia));
}

// From G = X^H X in P.Y: js = 2 when every pair is orthogonal to tol; else T
// in P.Yt and S in sigma.
__global__ void __launch_bounds__(512) k_jac_step(Dims* dims, const ProbPtr* __restrict__ ptrs, int cond, float tolu,
                                                  float small_u) {
  extern __shared__ __align__(16) unsigned char jp_raw[];
  __shared__ double s_n[JP_MAXL];
  __shared__ int s_k[JP_MAXL];  // S_c = 2^s_k
  __shared__ float red[16];
  const int p = blockIdx.x;
  const Dims D = dims[p];
  if (!jp_takes(D, cond) || D.js != 1) return;
  const ProbPtr P = ptrs[p];
  const int L = D.l, tid = threadIdx.x;
  const cplx* G = P.Y;
  float2* K = reinterpret_cast<float2*>(jp_raw);  // K[b * L + a] = K_ab
  __shared__ double s_f2;
  jp_scales(G, L, small_u, s_n, s_k, &s_f2);
  const double small = s_f2;
  float worst = 0.f;
  for (int i = tid; i < L * L; i += 512) {
    const int a = i % L, b = i / L;
    if (a == b) K[i] = make_float2(0.f, 0.f);
    if (a >= b) continue;
    const float2 k = jp_angle(G[(size_t)b * L + a], s_n[a], s_n[b], s_k[a], s_k[b], small, worst);
    K[i] = k;                                  // K_ab = t e
    K[a * L + b] = make_float2(-k.x, k.y);     // K_ba = -conj
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const float y = __shfl_xor_sync(0xffffffffu, worst, o);
    worst = (y > worst || y != y) ? y : worst;
  }
  if ((tid & 31) == 0) red[tid >> 5] = worst;
  __syncthreads();
  worst = 0.f;
  for (int w = 0; w < 16; ++w) worst = (red[w] > worst || red[w] != red[w]) ? red[w] : worst;
  if (worst <= tolu * sqrtf((float)L)) {
    if (tid == 0) dims[p].js = 2;
    return;
  }
  for (int i = tid; i < L * L; i += 512) {
    const int a = i % L, b = i / L;
    float sx = 0.f, sy = 0.f;
    for (int k = 0; k < L; ++k) {
      const float2 u = K[k * L + a], v = K[b * L + k];
      sx = fmaf(u.x, v.x, fmaf(-u.y, v.y, sx));
      sy = fmaf(u.x, v.y, fmaf(u.y, v.x, sy));
    }
    const float2 k1 = K[i];
    P.Yt[i] = cmk((a == b ? 1.0 : 0.0) + (double)k1.x + 0.5 * (double)sx, (double)k1.y + 0.5 * (double)sy);
  }
  for (int c = tid; c < L; c += 512) P.sigma[c] = __longlong_as_double((long long)(1023 + s_k[c]) << 52);
}

// ---------------------------------------------------------------------------
// l in (JP_MAXL, JB_MAXL]: the FP32 matrices no longer fit one SM.  A cluster
// of eight CTAs per problem, a warp per pair with the pair's columns in its
// registers, X and J in global memory and exchanged through L2 as in
// k_jacobi_cl.  Bound by the latency of a round (two trips to L2 and a cluster
// barrier).  Measured: 15 problems of l up to 266 4.7 ms (with the corrections
// and the check 15 ms; the FP64 cluster kernel alone took 62), 8 of l = 200
// 1.8 ms (22 ms).
// ---------------------------------------------------------------------------
enum { JB_MAXL = 320, JB_CL = 8, JB_ROWS = JB_MAXL / 32, JB_THREADS = JB_MAXL / 2 / JB_CL * 32 };

__global__ void __cluster_dims__(JB_CL, 1, 1) __launch_bounds__(JB_THREADS)
    k_jac_pre_cl(Dims* dims, const ProbPtr* __restrict__ ptrs, float2* scr, size_t stride, int cond) {
  __shared__ int s_exp;
  __shared__ int rotated;
  cg::cluster_group cluster = cg::this_cluster();
  const int crank = (int)cluster.block_rank(), p = blockIdx.x / JB_CL;
  const Dims D = dims[p];
  if (!jp_takes(D, cond)) {  // uniform over the cluster
    if ((cond & DPC_WIDE) && crank == 0 && threadIdx.x == 0) dims[p].js = 0;
    return;
  }
  const ProbPtr P = ptrs[p];
  const int L = D.l, tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, warp = tid >> 5, nw = nt >> 5;
  float2* X = scr + (size_t)p * stride;
  float2* J = X + (size_t)L * L;
  float* nrm = reinterpret_cast<float*>(P.sigma);
  if (tid == 0) s_exp = 0;
  __syncthreads();
  int e = 0;
  bool bad = false;
  for (int i = tid; i < L * L; i += nt) {
    const cplx v = P.R[i];
    e = max(e, max(oz_exp(v.x), oz_exp(v.y)));
    bad |= !isfinite(v.x) || !isfinite(v.y);
  }
  atomicMax(&s_exp, e);
  const bool any_bad = __syncthreads_or(bad);
  const int E = s_exp;
  if (any_bad || E == 0) {  // left to the Jacobi kernels as it is
    if (crank == 0 && tid == 0) dims[p].js = 0;
    return;
  }
  const int up = 1023 - E;
  for (int i = crank * nt + tid; i < L * L; i += JB_CL * nt) {
    const cplx v = P.R[i];
    X[i] = make_float2(jp_f32(v.x, up), jp_f32(v.y, up));
    J[i] = make_float2((i / L) == (i % L) ? 1.f : 0.f, 0.f);
  }
  cluster.sync();
  const int gw = warp * JB_CL + crank, nga = nw * JB_CL;  // warps over the cluster, interleaved
  const int Lp = (L + 1) & ~1;
  for (int sweep = 0; sweep < JP_SWEEPS; ++sweep) {
    for (int c = gw; c < L; c += nga) {
      float s = 0.f;
      for (int r = lane; r < L; r += 32) {
        const float2 v = __ldcg(X + (size_t)c * L + r);
        s = fmaf(v.x, v.x, fmaf(v.y, v.y, s));
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
      if (lane == 0) nrm[c] = s;
    }
    if (tid == 0) rotated = 0;
    cluster.sync();
    for (int rnd = 0; rnd < Lp - 1; ++rnd) {
      for (int pi = gw; pi < Lp / 2; pi += nga) {
        int a = pi == 0 ? Lp - 1 : rnd + pi, b = pi == 0 ? rnd : rnd - pi;
        if (pi > 0) {
          if (a >= Lp - 1) a -= Lp - 1;
          if (b < 0) b += Lp - 1;
        }
        if (a > b) {
          const int t = a;
          a = b;
          b = t;
        }
        if (b >= L) continue;  // uniform over the warp
        float2* xa = X + (size_t)a * L;
        float2* xb = X + (size_t)b * L;
        const float na = __ldcg(nrm + a), nb = __ldcg(nrm + b);
        float2 u[JB_ROWS], v[JB_ROWS];
#pragma unroll
        for (int q = 0; q < JB_ROWS; ++q) {
          const int r = lane + 32 * q;
          u[q] = r < L ? __ldcg(xa + r) : make_float2(0.f, 0.f);
          v[q] = r < L ? __ldcg(xb + r) : make_float2(0.f, 0.f);
        }
        if (!(na > 1e-34f) || !(nb > 1e-34f)) continue;  // below FP32's squares
        float gx = 0.f, gy = 0.f;
#pragma unroll
        for (int q = 0; q < JB_ROWS; ++q) {
          gx = fmaf(u[q].x, v[q].x, fmaf(u[q].y, v[q].y, gx));
          gy = fmaf(u[q].x, v[q].y, fmaf(-u[q].y, v[q].x, gy));
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
          gx += __shfl_xor_sync(0xffffffffu, gx, o);
          gy += __shfl_xor_sync(0xffffffffu, gy, o);
        }
        JpRot R;
        if (!jp_rotation(na, nb, gx, gy, R)) continue;
#pragma unroll
        for (int q = 0; q < JB_ROWS; ++q) {
          const int r = lane + 32 * q;
          if (r < L) jp_rotate(R, u[q], v[q], xa[r], xb[r]);
        }
        float2* ja = J + (size_t)a * L;
        float2* jb = J + (size_t)b * L;
#pragma unroll
        for (int q = 0; q < JB_ROWS; ++q) {
          const int r = lane + 32 * q;
          u[q] = r < L ? __ldcg(ja + r) : make_float2(0.f, 0.f);
          v[q] = r < L ? __ldcg(jb + r) : make_float2(0.f, 0.f);
        }
#pragma unroll
        for (int q = 0; q < JB_ROWS; ++q) {
          const int r = lane + 32 * q;
          if (r < L) jp_rotate(R, u[q], v[q], ja[r], jb[r]);
        }
        if (lane == 0) {
          nrm[a] = fmaxf(na - R.tg, 0.f);
          nrm[b] = nb + R.tg;
          rotated = 1;
        }
      }
      cluster.sync();  // the round's columns and norms visible to the cluster
    }
    int any = 0;
    for (int r = 0; r < JB_CL; ++r) any |= *cluster.map_shared_rank(&rotated, r);
    cluster.sync();  // every CTA has read the flags before they are reset
    if (!any) break;
  }
  for (int i = crank * nt + tid; i < L * L; i += JB_CL * nt) {
    const float2 v = __ldcg(J + i);
    P.J[i] = cmk((double)v.x, (double)v.y);
  }
  // S from the columns of X itself
  for (int c = gw; c < L; c += nga) {
    int m = 0;
    for (int r = lane; r < L; r += 32) {
      const cplx v = P.R[(size_t)c * L + r];
      m = max(m, max(oz_exp(v.x), oz_exp(v.y)));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
    if (lane == 0) P.sigma[c] = m > 0 ? __longlong_as_double((long long)max(1, 2046 - m) << 52) : 1.0;
  }
  if (crank == 0 && tid == 0) dims[p].js = 1;
}

// k_jac_step's K for l above JP_MAXL, into the scratch; a CTA takes JK_COLS
// columns and leaves its largest cosine in worst[p] (bits of a non-negative
// float, NaN the largest; zero before the launch).
enum { JK_COLS = 16 };

__global__ void __launch_bounds__(256) k_jac_k(const Dims* __restrict__ dims, const ProbPtr* __restrict__ ptrs,
                                               float2* scr, size_t stride, unsigned* worst_out, int cond,
                                               float small_u) {
  __shared__ double s_n[JB_MAXL];
  __shared__ int s_k[JB_MAXL];
  __shared__ double s_f2;
  const int p = blockIdx.y;
  const Dims D = dims[p];
  const int L = D.l, tid = threadIdx.x, c0 = blockIdx.x * JK_COLS;
  if (!jp_takes(D, cond) || D.js != 1 || c0 >= L) return;
  const ProbPtr P = ptrs[p];
  const cplx* G = P.Y;
  float2* K = scr + (size_t)p * stride;
  jp_scales(G, L, small_u, s_n, s_k, &s_f2);
  const double small = s_f2;
  float worst = 0.f;
  for (int i = tid; i < L * JK_COLS; i += 256) {
    const int r = i % L, c = c0 + i / L;
    if (c >= L) continue;
    const int a = min(r, c), b = max(r, c);
    float2 k = make_float2(0.f, 0.f);
    if (a != b) k = jp_angle(G[(size_t)b * L + a], s_n[a], s_n[b], s_k[a], s_k[b], small, worst);
    K[(size_t)c * L + r] = r < c ? k : make_float2(-k.x, k.y);  // K_ab = t e, K_ba = -conj
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const float y = __shfl_xor_sync(0xffffffffu, worst, o);
    worst = (y > worst || y != y) ? y : worst;
  }
  if ((tid & 31) == 0) atomicMax(worst_out + p, __float_as_uint(worst) & 0x7FFFFFFFu);
  if (blockIdx.x == 0)
    for (int c = tid; c < L; c += 256) P.sigma[c] = __longlong_as_double((long long)(1023 + s_k[c]) << 52);
}

__global__ void k_jac_done(Dims* dims, const unsigned* __restrict__ worst, int batch, float tolu) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p < batch && dims[p].js == 1 && __uint_as_float(worst[p]) <= tolu * sqrtf((float)dims[p].l)) dims[p].js = 2;
}

// T = I + K + K^2 / 2 in P.Yt, 32 x 32 per CTA.
__global__ void __launch_bounds__(256) k_jac_t(const Dims* __restrict__ dims, const ProbPtr* __restrict__ ptrs,
                                               const float2* scr, size_t stride, int cond) {
  __shared__ float2 A[32][33], Bt[32][33];  // [k][a], [b][k]
  const int p = blockIdx.z;
  const Dims D = dims[p];
  const int L = D.l, a0 = blockIdx.x * 32, b0 = blockIdx.y * 32;
  if (!jp_takes(D, cond) || D.js != 1 || a0 >= L || b0 >= L) return;
  const float2* K = scr + (size_t)p * stride;
  const int tid = threadIdx.x, lane = tid & 31, ty = tid >> 5;
  float2 acc[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) acc[q] = make_float2(0.f, 0.f);
  for (int k0 = 0; k0 < L; k0 += 32) {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int y = ty + 8 * q;
      A[y][lane] = (k0 + y < L && a0 + lane < L) ? K[(size_t)(k0 + y) * L + a0 + lane] : make_float2(0.f, 0.f);
      Bt[y][lane] = (b0 + y < L && k0 + lane < L) ? K[(size_t)(b0 + y) * L + k0 + lane] : make_float2(0.f, 0.f);
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
      const float2 k1 = K[(size_t)b * L + a];
      ptrs[p].Yt[(size_t)b * L + a] =
          cmk((a == b ? 1.0 : 0.0) + (double)k1.x + 0.5 * (double)acc[q].x, (double)k1.y + 0.5 * (double)acc[q].y);
    }
  }
}

cudaError_t jac_pre_prepare() {
  static DeviceOnce once;
  return once([] {
    const int b = (int)(sizeof(float2) * JP_MAXL * JP_MAXL);
    const cudaError_t e = cudaFuncSetAttribute(k_jac_pre, cudaFuncAttributeMaxDynamicSharedMemorySize, b);
    return e != cudaSuccess ? e : cudaFuncSetAttribute(k_jac_step, cudaFuncAttributeMaxDynamicSharedMemorySize, b);
  });
}

__global__ void k_jac_none(Dims* dims, int batch) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p < batch) dims[p].js = 0;
}

cudaError_t launch_jac_none(Dims* dims, int batch, cudaStream_t st) {
  k_jac_none<<<(batch + 127) / 128, 128, 0, st>>>(dims, batch);
  return cudaGetLastError();
}

bool jac_pre_rule(const Caps& cap, bool whole) { return cap.l <= JP_MAXL || (whole && cap.l <= JB_MAXL); }

#define JP_TRY(x)                     \
  do {                                \
    cudaError_t e_ = (x);             \
    if (e_ != cudaSuccess) return e_; \
  } while (0)

cudaError_t run_jac_pre(Dims* dims, const ProbPtr* ptrs, int batch, const Caps& cap, const OzScratch& oz, int chunk,
                        int cond, bool fp64, int* err, cudaStream_t st) {
  JP_TRY(jac_pre_prepare());
  const bool big = cap.l > JP_MAXL;
  const size_t sm = big ? 0 : sizeof(float2) * (size_t)cap.l * cap.l;
  // scratch of the wide form: the digits of the products before and after (at
  // least 28 l n bytes a problem, of which it takes 16 l^2, and 4 more)
  float2* scr = reinterpret_cast<float2*>(oz.ad);
  const size_t stride = 2 * (size_t)cap.l * cap.l;
  unsigned* worst = reinterpret_cast<unsigned*>(scr + stride * batch);
  const int js = cond | DPC_JS;
  auto prod = [&](int stage) { return launch_oz_range(stage, dims, ptrs, batch, cap, oz, chunk, js, err, st); };
  {
    ProfScope ps("k_jacobi[pre]", st);
    if (big) {
      // a warp per pair over the cluster
      const int nw = ((cap.l + 1) / 2 + JB_CL - 1) / JB_CL;
      k_jac_pre_cl<<<batch * JB_CL, nw * 32, 0, st>>>(dims, ptrs, scr, stride, cond);
    } else {
      // a group per pair where that takes at most JP_THREADS threads
      const int nt = ((cap.l + 1) / 2 * JP_G + 31) / 32 * 32;
      k_jac_pre<<<batch, nt < 128 ? 128 : (nt > JP_THREADS ? JP_THREADS : nt), sm, st>>>(dims, ptrs, cond);
    }
    JP_TRY(cudaGetLastError());
  }
  for (int it = 0; it < 2; ++it) {  // |E| ~ 1e-6, then its cube
    JP_TRY(prod(G_JG));                                           // J^H J = I + E
    JP_TRY(launch_lowdin_j(dims, ptrs, batch, cap.l, cond, st));  // T = (J^H J)^-1/2
    JP_TRY(prod(G_JT));                                           // J <- J T
  }
  JP_TRY(prod(G_XJ));  // X <- X J
  // tolerances of the kernels that would go on: 4 eps sqrt(l) and L eps in
  // FP64, 8 2^-48 sqrt(l) and L 2^-48 in double-float
  const float tolu = fp64 ? 8.8817842e-16f : 2.8421709e-14f, small_u = fp64 ? 2.220446e-16f : 3.5527137e-15f;
  for (int it = 0; it <= JP_STEPS; ++it) {
    JP_TRY(prod(G_XG));
    {
      ProfScope ps("k_jacobi[step]", st);
      if (big) {
        JP_TRY(cudaMemsetAsync(worst, 0, sizeof(unsigned) * batch, st));
        k_jac_k<<<dim3((cap.l + JK_COLS - 1) / JK_COLS, batch), 256, 0, st>>>(dims, ptrs, scr, stride, worst, cond,
                                                                              small_u);
        k_jac_done<<<(batch + 127) / 128, 128, 0, st>>>(dims, worst, batch, tolu);
        const int nb = (cap.l + 31) / 32;
        k_jac_t<<<dim3(nb, nb, batch), 256, 0, st>>>(dims, ptrs, scr, stride, cond);
      } else {
        k_jac_step<<<batch, 512, sm, st>>>(dims, ptrs, cond, tolu, small_u);
      }
      JP_TRY(cudaGetLastError());
    }
    if (it == JP_STEPS) break;
    JP_TRY(prod(G_XT));
    JP_TRY(prod(G_JT));
  }
  return cudaSuccess;
}

}  // namespace tg
