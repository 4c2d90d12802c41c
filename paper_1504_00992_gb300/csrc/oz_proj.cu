// FP64-accurate projection on the tensor cores (sm_103a tcgen05, BF16 slices).
//
// The step B = Q^H A of Section IV (after Alg. 1), in the mixed form with the
// FP32 basis Q_f and its re-orthonormalisation Q = Q_f (I + D): C = Q_f^H A
// (l x n) is formed from error-free slices of both operands; the factor I + D
// is applied to the l x l matrices after it (launch_fold_small, qr_blocked.cu).
//
// Slices (Ozaki's error-free splitting; Ozaki, Ogita, Oishi, Rump, Numer.
// Algorithms 59, 2012): every row i of the left operand and every column j of
// the right one is scaled by its own power of two (the exponent of its
// largest entry over all k) to a 56-bit integer N, |N| <= 2^55, rounded to
// nearest, and N is cut into OZ_S = 7 balanced base-256 digits, |d_t| <= 128
// (N = sum_t d_t 256^(7-t)), each an exact BF16 number.  A product of two
// digits is an integer of at most 2^14, and level L = t + u of the digit
// pairs sums at most L - 1 pairs x 2 real products x k of them, so over
// OZ_DRAIN = 64 k every level up to 8 stays below 128 * 7 * 2^14 < 2^24: the
// tensor core's FP32 sums are exact integers.  The epilogue reads the
// fourteen accumulators (C_r and C_i at levels 2 .. 8) after every 64 k and
// adds levels 2 .. 6 exactly, in one 64-bit integer (moved to FP64 every 2^14
// k), and levels 7 and 8 (2^-40 and 2^-48 of the leading level) in one FP32
// number.  The scales are applied once at the end.  What is lost, in units of
// max|a| max|b| over the row and column: the rounding of the operands and the
// digit pairs with t + u > 8 (2^-56 each per k, random signs), and the FP32
// additions, K / 64 of them at 2^-24 of a sum below 2^-36 K: at most
// K^2 2^-67 (2^-56 K at K = 2000, 2^-54 K at K = 8000).  On a CPU emulation 1.8e-16
// relative at K = 64 and 3e-16 at K = 2000 for Gaussian or orthonormal
// operands, against 3e-16 and 1.5e-15 of FP64 multiply-adds in order; rows
// graded over 2^-46 give 1.4e-15 against 2e-15.  Six digits would give
// 4e-14 to 8e-14, eight would cost 36 digit pairs instead of 28 for accuracy
// FP64 results cannot hold.
//
// What bounds it.  An MMA of M = 128 costs ~130 cycles whatever its N up to 256
// (timed with every N set to 32: 10% less), so the 28 MMAs of a k step of 16
// are ~3600 cycles, and the 72 KB of digits of a k step take about as long at
// the 38 GB/s per SM the copies reach alone.  Tensor memory holds no wider
// tile than 32 columns of fourteen sums.  At 16 x 2000 x 2000 x 120 a product
// takes 1.6 ms (38 TFLOP/s FP64-equivalent; the FP64 pipe 54 ms), the read-out
// of the accumulators (which nothing overlaps) 0.35 ms of it.  Tried and not
// kept: reading out C_r while C_i is filled (stages held longer: 15% slower),
// clusters sharing the left operand by multicast (same time), TMA tiles (32-
// byte rows: 10% slower).
//
// Complex products: C_r = Ar Br - Ai Bi, C_i = Ar Bi + Ai Br with Ar, Ai the
// digits of Re and Im of the left operand and Br, Bi those of the right one;
// minus signs, and the conjugate of either operand, are the MMA's negate-A bit.
//
// The same kernel serves the other FP64-accurate products of the mixed form
// (k_oz_gemm<stage>): the Cholesky QR of B^H (Gram matrices B B^H and
// Q1^H Q1, the triangular products B^H R1^-1 and Q1 R2^-1, and B Qb) and
// U = Q J_k, V = Qb W_k.  Their operands are FP64 (the stage table of
// stages.cuh gives the layout); k_oz_digits_op cuts them into the same
// digits, and a conjugated left operand flips the negate bits of the MMAs
// that take its imaginary digits instead of negating them.
//
// Kernel structure (one CTA = 128 rows of C x OZ_BN = 32 columns, all k):
// warp 0 streams the digit planes of each 16-deep k step with bulk copies
// (the digit arrays are stored step by step, swizzled for the MMAs) into a
// ring of stages; warp 1 issues 28 tcgen05.mma.kind::f16 per k step:
// the digit planes u = 1 .. 7 of a part of B's side lie one after another in
// shared memory and the accumulators of levels 2 .. 8 one after another in
// tensor memory, so digit t of the other operand times planes 1 .. 8 - t is
// one MMA of N = 32 (8 - t) into the accumulators of levels t + 1 .. 8; warps
// 2 .. 17 read the accumulators after each 64 k (warp w reads TMEM lanes
// 32 (w % 4) .. +31 and a quarter of the columns) and keep the sums.  Every
// mbarrier wait is bounded; on expiry the kernel raises *err, waits for its
// own copies and MMAs, and frees its tensor memory.
#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <mutex>

#include "../../include/tebd_gb300.h"
#include "dfsplit.cuh"
#include "internal.cuh"
#include "mixed.cuh"
#include "once.cuh"
#include "profiler.cuh"
#include "stages.cuh"
#include "tc_sync.cuh"
#include "workspace.cuh"

namespace tg {

enum {
  OZ_S = 7,        // digits per operand
  OZ_KB = 64,      // k padding of the digit arrays
  OZ_KS = 16,      // k per MMA / TMA stage
  OZ_BM = 128,     // rows of C per CTA (TMEM lanes)
  OZ_BN = 32,      // columns of C per CTA
  OZ_DRAIN = 64,   // k per exact accumulation (the accumulators are read and cleared after each)
  OZ_SQ = 4,       // digits of the FP32 basis Q_f (of a theta whose rows are not graded)
  OZ_EPI_WARPS = 16,  // four per TMEM lane quadrant, 8 columns each
  OZ_THREADS = 64 + 32 * OZ_EPI_WARPS,
  OZ_NGRP = OZ_S,  // accumulators per part: levels 2 .. 8
  OZ_TMEM_COLS = 512,  // fourteen 32-column accumulators, rounded up to a power of two
  OZ_FLUSH = 256,  // blocks after which the integer sums move to FP64 (level 2: below 2^53 per block)
  OZ_SELF_K = 512  // depths up to this: the digit kernels find a row's largest exponent themselves
};

static const uint32_t OZ_A_TILE = OZ_BM * OZ_KS * 2;  // one digit tile of the left operand: 4 KB
static const uint32_t OZ_B_TILE = OZ_BN * OZ_KS * 2;  // one digit tile of the right operand: 1 KB

// ---------------------------------------------------------------------------
// Digits of one value relative to its row's largest biased FP64 exponent E:
// N = rint(x 2^(54 - (E - 1023))) with integer operations only (the FP64 pipe
// runs at 1/64 of the FP32 rate), then balanced base-256 digits: adding 128
// to each of the six lower digits makes them plain bytes.
// ---------------------------------------------------------------------------
// (shift: of x 2^shift)
__device__ __forceinline__ int64_t oz_fix(double x, int E, int shift) {
  const uint64_t u = (uint64_t)__double_as_longlong(x);
  const int e = (int)((u >> 52) & 0x7FF);
  if (e == 0 || e == 0x7FF) return 0;
  const int64_t m = (int64_t)((u & 0xFFFFFFFFFFFFFull) | (1ull << 52));
  const int sh = E - (e + shift) - 2;  // x = m 2^(e - 1075), N = m 2^-sh; sh >= -2
  const int64_t n = sh <= 0 ? (m << (-sh)) : (sh >= 56 ? 0 : ((m + (1ll << (sh - 1))) >> sh));
  return (u >> 63) ? -n : n;
}
// The same of an FP32 value for NS = 7 digits; for four, N = rint(x 2^(30 - (E - 1023))),
// |N| < 2^31 (E the row's largest exponent)
template <int NS>
__device__ __forceinline__ int64_t oz_fix_f32(float x, int E) {
  const unsigned u = __float_as_uint(x);
  const int e = (int)((u >> 23) & 0xFF);
  if (e == 0 || e == 0xFF) return 0;
  const int m = (int)((u & 0x7FFFFFu) | 0x800000u);
  if constexpr (NS == OZ_SQ) {
    const int sh = E - (e - 127 + 1023) - 7;  // x = m 2^(e - 150), N = m 2^-sh; sh >= -7
    const int n = sh <= 0 ? (m << (-sh)) : (sh >= 26 ? 0 : ((m + (1 << (sh - 1))) >> sh));
    return (u >> 31) ? -n : n;
  }
  const int sh = E - (e - 127 + 1023) - 31;  // sh >= -31
  const int64_t n = sh <= 0 ? ((int64_t)m << (-sh)) : (sh >= 26 ? 0 : ((m + (1 << (sh - 1))) >> sh));
  return (u >> 31) ? -n : n;
}

// The NS digits of four values of 8 NS bits as packed BF16 quadruples (planes t = 1 .. NS).
template <int NS>
__device__ __forceinline__ void oz_digits4(const int64_t n[4], uint2 d[NS]) {
  const float bias = 8388608.f + 128.f;
  uint64_t m[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) m[q] = (uint64_t)n[q] + (0x0000808080808080ull >> (8 * (OZ_S - NS)));
#pragma unroll
  for (int t = 0; t < NS; ++t) {
    unsigned f[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      if (t == 0)
        f[q] = __float_as_uint((float)(int)((int64_t)m[q] >> (8 * (NS - 1))));
      else
        f[q] = __float_as_uint(__uint_as_float(0x4B000000u | (unsigned)((m[q] >> (8 * (NS - 1 - t))) & 0xFF)) - bias);
    }
    d[t].x = __byte_perm(f[0], f[1], 0x7632);  // the upper halves: exact BF16 numbers
    d[t].y = __byte_perm(f[2], f[3], 0x7632);
  }
}

// Where a digit lives: [z][k step][plane][row][16 k], 32 bytes per row and
// step, so that the rows of a tile are one run per plane (a bulk copy each)
// and lie in shared memory as the MMA's 32-byte swizzle wants them: the two
// 16-byte halves of a row trade places where bit 2 of the row is set.
// Offset in digits of the half `ch` (k 8 ch .. 8 ch + 7) of k step ks.
template <int NS>
__device__ __forceinline__ size_t oz_at(int ks, int plane, int row, int ch, int rc) {
  return (((size_t)ks * (2 * NS) + plane) * rc + row) * OZ_KS + 8 * (ch ^ ((row >> 2) & 1));
}

// Scale of a row in the product: 2^(E - 1023 - 22); zero for a zero row, NaN
// for a row with a non-finite entry (whose digits are zero): the row or column
// of the result is NaN then, as a sum of FP64 multiply-adds would make it.
__device__ __forceinline__ double oz_scale(int E) {
  if (E == OZ_NONFINITE) return __longlong_as_double(0x7FF8ll << 48);
  return E > 22 ? __longlong_as_double((long long)(E - 22) << 52) : 0.0;
}

// ---------------------------------------------------------------------------
// Stages.  OZ_PROJ is the projection C = Q_f^H A (l x n, K = m), written as
// C^H = A^H Q_f into Yt; the others are the GemmStage products of stages.cuh,
// C = op(A) op(B) with op(A) conjugated where StageFlags says so and C
// stored conjugated for G_V.
// ---------------------------------------------------------------------------
// OZ_THETA, OZ_GATE: the contraction and the gate of bonds whose gate is a
// GEMM (d_l d_r >= GATE_GEMM_MIN), the mixed forms' counterparts of
// k_cgemm_df<DgTheta> / <DgGate> (df_gemm.cu documents the operands).
// OZ_GRAMY, OZ_GRAMT: Gram matrices of FP32 sketches (m or n rows), as OZ_GRAM
// but without subtracting the identity.
// OZ_PROJ7, OZ_GRAM7: OZ_PROJ and OZ_GRAM of the instances whose Q_f takes seven
// digits (Dims::gr).
enum { OZ_PROJ = 100, OZ_GRAM = 101, OZ_THETA = 102, OZ_GATE = 103, OZ_GRAMY = 104, OZ_GRAMT = 105,
       OZ_PROJ7 = 107, OZ_GRAM7 = 108,
       OZ_CONT = 106 };  // OZ_THETA for the bonds of theta_digits_rule without a pre-gate buffer, into theta
template <int ST>
struct OzFp32Gram {
  static constexpr bool yes = ST == OZ_GRAM || ST == OZ_GRAM7 || ST == OZ_GRAMY || ST == OZ_GRAMT;
};
template <int ST>
struct OzProj {
  static constexpr bool yes = ST == OZ_PROJ || ST == OZ_PROJ7;
};
static_assert(OZ_THETA == OZ_THETA_STAGE && OZ_GATE == OZ_GATE_STAGE && OZ_CONT == OZ_CONT_STAGE,
              "stage ids of mixed.cuh");

struct OzOp {
  int M, N, K;  // rows and columns of C, depth
  cplx* C;
  int64_t crs, ccs;
};

template <int ST>
__device__ __forceinline__ OzOp oz_op(const Dims& D, const ProbPtr& P) {
  OzOp o;
  if constexpr (OzProj<ST>::yes) {
    o.M = D.l; o.N = D.n; o.K = D.m;
    o.C = P.Yt; o.crs = D.n; o.ccs = 1;  // element (j, i) of the n x l column-major B^H
  } else if constexpr (OzFp32Gram<ST>::yes) {
    o.M = D.l; o.N = D.l; o.K = ST == OZ_GRAMT ? D.n : D.m;
    o.C = P.R; o.crs = 1; o.ccs = D.l;  // OZ_GRAM: E = Q_f^H Q_f - I; l x l column-major
  } else if constexpr (ST == OZ_THETA || ST == OZ_CONT) {
    o.M = D.dl * D.cl; o.N = D.dr * D.cr; o.K = D.cm;  // into the pre-gate buffer or theta (oz_store)
    o.C = ST == OZ_THETA ? P.Cpre : const_cast<cplx*>(P.theta); o.crs = D.n; o.ccs = 1;
  } else if constexpr (ST == OZ_GATE) {
    o.M = D.dl * D.dr; o.N = D.cl * D.cr; o.K = D.dl * D.dr;  // into theta (oz_store)
    o.C = const_cast<cplx*>(P.theta); o.crs = 0; o.ccs = 0;
  } else {
    const GemmOp g = gemm_of<ST>(D, P);
    o.M = g.M; o.N = g.N; o.K = g.K;
    o.C = g.C; o.crs = g.crs; o.ccs = g.ccs;
  }
  return o;
}

template <int ST>
struct OzConj {
  static constexpr bool own = ST < OZ_PROJ;  // a GemmStage of stages.cuh
  static constexpr bool A = OzProj<ST>::yes || OzFp32Gram<ST>::yes || (own && StageFlags<ST>::conjA);  // Q_f^H
  static constexpr bool C = OzProj<ST>::yes || (own && StageFlags<ST>::conjC);
};

// Digits of each operand and the ring of stages of a product.
template <int ST>
struct OzGeo {
  static constexpr bool four = OzFp32Gram<ST>::yes && ST != OZ_GRAM7;
  static constexpr int SA = (ST == OZ_PROJ || four) ? OZ_SQ : OZ_S;
  static constexpr int SB = four ? OZ_SQ : OZ_S;
  static constexpr uint32_t A_STAGE = 2 * SA * OZ_A_TILE, B_STAGE = 2 * SB * OZ_B_TILE;
  static constexpr int STAGES = SA == OZ_S ? 3 : 4;
  static constexpr size_t smem = 1024 + (size_t)STAGES * (A_STAGE + B_STAGE) + (2 * STAGES + 3) * 8 + 16;
};

// The stages that skip a bond: the contraction and gate GEMMs run only for
// bonds with a pre-gate buffer.
template <int ST>
__device__ __forceinline__ bool oz_skip(const Dims& D, const ProbPtr& P) {
  if (ST == OZ_CONT) return P.Cpre != nullptr || !theta_digits_rule(D.m, D.n, D.cm);
  return (ST == OZ_THETA || ST == OZ_GATE) && P.Cpre == nullptr;
}

// Whether a launch's condition bits take a problem.
__device__ __forceinline__ bool oz_takes(const Dims& D, int cond) {
  if ((cond >> DPC_PASS) > 0 && D.cq < (cond >> DPC_PASS)) return false;
  if ((cond & DPC_OK) && D.cf) return false;
  if ((cond & DPC_QFLAG) && !D.qflag) return false;
  if ((cond & DPC_DIG) && !D.dig) return false;
  if ((cond & DPC_CHK) && !D.chk) return false;
  if ((cond & DPC_JS) && D.js != 1) return false;
  if ((cond & DPC_WIDE) && D.l < DP_WIDE_L) return false;
  if ((cond & DPC_GRADED) && !D.gr) return false;
  if ((cond & DPC_FLAT) && D.gr) return false;
  return true;
}

// Element (i, j) of C into its destination.
template <int ST>
__device__ __forceinline__ void oz_store(const Dims& D, const ProbPtr& P, const OzOp& op, int i, int j, double re,
                                         double im) {
  if constexpr (ST == OZ_THETA || ST == OZ_CONT) {
    // lam_l[alpha] lam_r[beta] scale the contraction (rows (i, alpha), columns (j, beta))
    op.C[(int64_t)i * D.n + j] = cscale(cmk(re, im), P.laml[i % D.cl] * P.lamr[j % D.cr]);
  } else if constexpr (ST == OZ_GATE) {
    const int a = i / D.dr, b = i - a * D.dr, al = j / D.cr, be = j - al * D.cr;  // rows (i, j), columns (alpha, beta)
    op.C[(int64_t)(a * D.cl + al) * D.n + b * D.cr + be] = cmk(re, im);
  } else {
    if ((ST == OZ_GRAM || ST == OZ_GRAM7) && i == j) re -= 1.0;  // E = Q_f^H Q_f - I
    op.C[(int64_t)i * op.crs + (int64_t)j * op.ccs] = cmk(re, OzConj<ST>::C ? -im : im);
  }
}

// 1 / x of a power of two
__device__ __forceinline__ double oz_pow2_inv(double x) {
  return __longlong_as_double((2046ll << 52) - __double_as_longlong(x));
}

// Operand sources of k_oz_digits_op in their K-major views: element (row, k)
// of side 0 (rows of op(A)) or side 1 (columns of op(B)), and whether
// consecutive rows are adjacent in memory (else consecutive k are).
template <int ST, int SIDE>
struct OzSrc {  // a GemmStage: strided operand of the stage table
  const cplx* X;
  const double* scale;
  int64_t rs, ks;
  int rows, K;
  __device__ OzSrc(const Dims& D, const ProbPtr& P) : scale(P.sigma) {
    const GemmOp g = gemm_of<ST>(D, P);
    rows = SIDE == 0 ? g.M : g.N;
    K = g.K;
    X = SIDE == 0 ? g.A : g.B;
    rs = SIDE == 0 ? g.ars : g.bcs;
    ks = SIDE == 0 ? g.acs : g.brs;
  }
  __device__ bool rows_contig() const { return rs == 1; }
  __device__ int shift(int) const { return 0; }
  __device__ cplx at(int r, int k) const {
    const cplx v = X[(int64_t)r * rs + (int64_t)k * ks];
    if constexpr (SIDE == 0 && StageFlags<ST>::scaleA) return cscale(v, scale[k]);
    if constexpr (SIDE == 1 && StageFlags<ST>::scaleB) return cscale(v, oz_pow2_inv(scale[k]));
    return v;
  }
};
template <>
struct OzSrc<OZ_PROJ, 1> {  // the columns of theta
  const cplx* X;
  int rows, K;
  __device__ OzSrc(const Dims& D, const ProbPtr& P) : X(P.theta), rows(D.n), K(D.m) {}
  __device__ bool rows_contig() const { return true; }
  __device__ int shift(int) const { return 0; }
  __device__ cplx at(int r, int k) const { return X[(int64_t)k * rows + r]; }
};
// The shifts of a bond's contraction (k_oz_balance), in the sketch matrix's
// buffer, which the truncation fills later; null for a bond whose buffer is
// shorter than chi_m.
__device__ __forceinline__ int* oz_shifts(const Dims& D, const ProbPtr& P) {
  return (int64_t)D.cm <= 4ll * D.n * D.l ? reinterpret_cast<int*>(P.omega) : nullptr;
}

template <int SIDE>
struct OzSrc<OZ_THETA, SIDE> {  // A = Gamma_l (rows (i, alpha)), B = lam_m Gamma_r (columns (j, beta))
  Dims D;
  const ProbPtr* P;
  const int* sh;
  int rows, K;
  __device__ OzSrc(const Dims& d, const ProbPtr& p) : D(d), P(&p), sh(oz_shifts(d, p)) {
    rows = SIDE == 0 ? d.dl * d.cl : d.dr * d.cr;
    K = d.cm;
  }
  __device__ bool rows_contig() const { return SIDE == 1; }
  __device__ int shift(int g) const { return (sh && g < K) ? (SIDE == 0 ? sh[g] : -sh[g]) : 0; }
  __device__ cplx at(int r, int g) const {
    if (SIDE == 0) {
      const int i = r / D.cl, al = r - i * D.cl;
      return P->gl[((int64_t)i * P->cap_l + al) * P->cap_m + g];
    }
    const int j = r / D.cr, be = r - j * D.cr;
    return cscale(P->gr[((int64_t)j * P->cap_m + g) * P->cap_r + be], P->lamm[g]);
  }
};
template <int SIDE>
struct OzSrc<OZ_CONT, SIDE> : OzSrc<OZ_THETA, SIDE> {
  __device__ OzSrc(const Dims& d, const ProbPtr& p) : OzSrc<OZ_THETA, SIDE>(d, p) {}
};
template <int SIDE>
struct OzSrc<OZ_GATE, SIDE> {  // A = the gate (rows (i, j)), B = the (i', j') x (alpha, beta) gather of C
  Dims D;
  const ProbPtr* P;
  int rows, K;
  __device__ OzSrc(const Dims& d, const ProbPtr& p) : D(d), P(&p) {
    rows = SIDE == 0 ? d.dl * d.dr : d.cl * d.cr;
    K = d.dl * d.dr;
  }
  __device__ bool rows_contig() const { return SIDE == 1; }
  __device__ int shift(int) const { return 0; }
  __device__ cplx at(int r, int k) const {
    if (SIDE == 0) return P->gate[(int64_t)r * (D.dl * D.dr) + k];
    const int ip = k / D.dr, jp = k - ip * D.dr, al = r / D.cr, be = r - al * D.cr;
    return P->Cpre[(int64_t)(ip * D.cl + al) * D.n + jp * D.cr + be];
  }
};

// Exponent of an entry times 2^shift.
__device__ __forceinline__ int oz_exp(cplx v, int shift) {
  const int e = max(oz_exp(v.x), oz_exp(v.y));
  return (e == 0 || e == OZ_NONFINITE) ? e : max(e + shift, 0);
}

// The contraction sum_g Gamma_l[., g] (lam_m[g] Gamma_r[g, .]) does not see a
// factor moved between the two sides of a term g, but digits relative to a
// row's largest entry do: a column of Gamma_l that is large where lam_m is
// small (1e14 at lam_m = 1e-14 in a gauge that is not canonical) left ten bits
// of the others.  So both sides of every term are brought to the same largest
// entry by a power of two: shift[g] is half the difference of the exponents,
// and only the exponents the digits are cut at change.  A CTA takes 32 terms,
// one read of both Gammas.
template <int ST>
__global__ void __launch_bounds__(256) k_oz_balance(const Dims* __restrict__ dims, const ProbPtr* __restrict__ ptrs,
                                                    int cond) {
  __shared__ int ea[32], eb[32];
  const int z = blockIdx.y;
  const Dims D = dims[z];
  if (!D.active || !oz_takes(D, cond) || oz_skip<ST>(D, ptrs[z])) return;
  const ProbPtr& P = ptrs[z];
  int* sh = oz_shifts(D, P);
  const int g0 = blockIdx.x * 32;
  if (!sh || g0 >= D.cm) return;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (tid < 32) ea[tid] = eb[tid] = 0;
  __syncthreads();
  int e = 0;
  if (g0 + lane < D.cm)
    for (int i = 0; i < D.dl; ++i) {
      const cplx* row = P.gl + (int64_t)i * P.cap_l * P.cap_m + g0 + lane;
#pragma unroll 4
      for (int al = warp; al < D.cl; al += 8) e = max(e, oz_exp(row[(int64_t)al * P.cap_m], 0));
    }
  atomicMax(&ea[lane], e);
  for (int q = warp; q < 32 && g0 + q < D.cm; q += 8) {
    e = 0;
    for (int j = 0; j < D.dr; ++j) {
      const cplx* row = P.gr + ((int64_t)j * P.cap_m + g0 + q) * P.cap_r;
#pragma unroll 4
      for (int be = lane; be < D.cr; be += 32) e = max(e, oz_exp(row[be], 0));
    }
    e = __reduce_max_sync(0xffffffffu, e);
    if (lane == 0) eb[q] = e;
  }
  __syncthreads();
  if (tid < 32 && g0 + tid < D.cm) {
    const int a = ea[tid], b = eb[tid], l = oz_exp(P.lamm[g0 + tid]);
    const bool any = a > 0 && b > 0 && l > 0 && a < OZ_NONFINITE && b < OZ_NONFINITE && l < OZ_NONFINITE;
    sh[g0 + tid] = any ? (b + l - 1023 - a) >> 1 : 0;
  }
}

// Largest biased exponent of every row of a stage operand into Es[z][row]
// (zero before the launch; a maximum does not depend on the order of the
// atomics).  A CTA takes 16 rows x OZ_MAX_K k.
enum { OZ_MAX_K = 512 };

template <int ST, int SIDE>
__global__ void __launch_bounds__(256) k_oz_max(const Dims* __restrict__ dims, const ProbPtr* __restrict__ ptrs,
                                                int* Es, int rc, int cond) {
  __shared__ int emax[16];
  const int z = blockIdx.z;
  const Dims D = dims[z];
  if (!D.active || !oz_takes(D, cond) || oz_skip<ST>(D, ptrs[z])) return;
  const OzSrc<ST, SIDE> src(D, ptrs[z]);
  const int r0 = blockIdx.x * 16, k0 = blockIdx.y * OZ_MAX_K, k1 = min(src.K, k0 + OZ_MAX_K);
  if (r0 >= src.rows || k0 >= src.K) return;  // uniform over the block
  const int tid = threadIdx.x;
  if (tid < 16) emax[tid] = 0;
  __syncthreads();
  const bool rowc = src.rows_contig();
  int E = 0;
  int r;
  if (rowc) {
    r = tid & 15;
    if (r0 + r < src.rows)
      for (int k = k0 + (tid >> 4); k < k1; k += 16) E = max(E, oz_exp(src.at(r0 + r, k), src.shift(k)));
  } else {
    r = tid >> 4;
    if (r0 + r < src.rows)
      for (int k = k0 + (tid & 15); k < k1; k += 16) E = max(E, oz_exp(src.at(r0 + r, k), src.shift(k)));
  }
  atomicMax(&emax[r], E);
  __syncthreads();
  if (tid < 16 && r0 + tid < src.rows) atomicMax(&Es[(size_t)z * rc + r0 + tid], emax[tid]);
}

// Digits of a stage operand in its K-major view: SIDE 0 the rows i of op(A)
// (element A[i ars + k acs], not conjugated: the MMAs conjugate), SIDE 1 the
// columns j of op(B) (element B[k brs + j bcs]); into Xd (oz_at; rows rc, Kp / 16 k steps).  SELF: the CTA takes 16 rows and all k, finds their
// largest exponents itself (a second read of at most OZ_SELF_K k, from L2)
// and stores them; otherwise it takes 16 rows x 64 k and reads them from Es.
// Rows and k past the instance's own extents become zero digits.
struct OzDigSmem {
  cplx tile[16][OZ_KB + 1];
  __align__(16) uint16_t dig[2 * OZ_S][16][OZ_KB + 8];  // [reim t][row][k]
  int emax[16];
};

template <int ST, int SIDE, bool SELF>
__device__ __forceinline__ void oz_digits_block(const Dims* __restrict__ dims, const ProbPtr* __restrict__ ptrs,
                                                uint16_t* Xd, int* Es, int rc, int Kp, int cond, OzDigSmem& sm) {
  auto& tile = sm.tile;
  auto& dig = sm.dig;
  auto& emax = sm.emax;
  const int z = blockIdx.z;
  const Dims D = dims[z];
  if (!D.active || !oz_takes(D, cond) || oz_skip<ST>(D, ptrs[z])) return;
  const OzSrc<ST, SIDE> src(D, ptrs[z]);
  const int rows = src.rows, K = src.K;
  const bool rowc = src.rows_contig();
  const int r0 = blockIdx.x * 16;
  const int tid = threadIdx.x;
  const int r = tid >> 4, pq = tid & 15;  // 16 threads per row, 4 k each
  int E = 0;
  if (SELF) {
    if (tid < 16) emax[tid] = 0;
    __syncthreads();
    const int lr = rowc ? (tid & 15) : (tid >> 4);
    int e = 0;
    if (r0 + lr < rows)
      for (int k = rowc ? (tid >> 4) : (tid & 15); k < K; k += 16) e = max(e, oz_exp(src.at(r0 + lr, k), src.shift(k)));
    atomicMax(&emax[lr], e);
    __syncthreads();
    E = emax[r];
    if (pq == 0 && r0 + r < rc) Es[(size_t)z * rc + r0 + r] = E;
  } else {
    E = (r0 + r < rc) ? Es[(size_t)z * rc + r0 + r] : 0;
  }
  uint16_t* base = Xd + (size_t)z * 2 * OZ_S * rc * Kp;
  // whole blocks of 64 k the GEMM reads: zero digits past K within the last
  const int kend = min(Kp, ((K + OZ_KB - 1) / OZ_KB) * OZ_KB);
  for (int k0 = SELF ? 0 : (int)blockIdx.y * OZ_KB; k0 < kend; k0 += SELF ? OZ_KB : kend) {
    for (int e = tid; e < 16 * OZ_KB; e += 256) {
      int tr, k;  // consecutive threads along the unit-stride direction
      if (rowc) { tr = e & 15; k = e >> 4; } else { k = e & (OZ_KB - 1); tr = e >> 6; }
      const int gr = r0 + tr, gk = k0 + k;
      tile[tr][k] = (gr < rows && gk < K) ? src.at(gr, gk) : cmk(0.0, 0.0);
    }
    __syncthreads();
    int64_t nr[4], ni[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const cplx v = tile[r][pq * 4 + q];
      const int sh = src.shift(k0 + pq * 4 + q);
      nr[q] = oz_fix(v.x, E, sh);
      ni[q] = oz_fix(v.y, E, sh);
    }
    uint2 d[OZ_S];
    oz_digits4<OZ_S>(nr, d);
#pragma unroll
    for (int t = 0; t < OZ_S; ++t) *reinterpret_cast<uint2*>(&dig[t][r][pq * 4]) = d[t];
    oz_digits4<OZ_S>(ni, d);
#pragma unroll
    for (int t = 0; t < OZ_S; ++t) *reinterpret_cast<uint2*>(&dig[OZ_S + t][r][pq * 4]) = d[t];
    __syncthreads();
    // (k step, plane, row, half) of 16 bytes each: 512-byte runs of 16 rows
    for (int w = tid; w < 2 * OZ_S * 16 * 8; w += 256) {
      const int ch = w & 1, rr = (w >> 1) & 15, t = w >> 5;  // t = plane + 14 k step
      const int plane = t % (2 * OZ_S), ks = t / (2 * OZ_S);
      if (r0 + rr >= rc) continue;
      *reinterpret_cast<uint4*>(base + oz_at<OZ_S>((k0 >> 4) + ks, plane, r0 + rr, ch, rc)) =
          *reinterpret_cast<const uint4*>(&dig[plane][rr][16 * ks + 8 * ch]);
    }
    if (SELF) __syncthreads();
  }
}

template <int ST, int SIDE, bool SELF>
__global__ void __launch_bounds__(256) k_oz_digits_op(const Dims* __restrict__ dims, const ProbPtr* __restrict__ ptrs,
                                                      uint16_t* Xd, int* Es, int rc, int Kp, int cond) {
  __shared__ OzDigSmem sm;
  oz_digits_block<ST, SIDE, SELF>(dims, ptrs, Xd, Es, rc, Kp, cond, sm);
}

// Both operands of a product in one launch (depths up to OZ_SELF_K).
template <int ST>
__global__ void __launch_bounds__(256) k_oz_digits_two(const Dims* __restrict__ dims, const ProbPtr* __restrict__ ptrs,
                                                       uint16_t* Ad, int* As, int ac, uint16_t* Bd, int* Bs, int bc,
                                                       int Kp, int cond) {
  __shared__ OzDigSmem sm;
  if (blockIdx.y == 0) {
    if ((int)blockIdx.x * 16 < ac) oz_digits_block<ST, 0, true>(dims, ptrs, Ad, As, ac, Kp, cond, sm);
  } else {
    if ((int)blockIdx.x * 16 < bc) oz_digits_block<ST, 1, true>(dims, ptrs, Bd, Bs, bc, Kp, cond, sm);
  }
}

// Digits of Q_f (m x l column-major FP32 complex per instance, capacity
// mc x lc) into Ad (oz_at) and Es[z][i]: one warp per column.  An FP32 column
// is four digits: its entries are rounded to multiples of 2^-31 of the power
// of two above the largest one, in place, so that every later use of Q_f sees
// the numbers the digits hold exactly (entries above 2^-8 of the largest one
// keep all their 24 bits).  Against seven digits the projection loads 47 KB
// instead of 72 KB per k step and runs 22 digit pairs instead of 28.  The same
// numbers go to P.Q in FP64, the left operand of U = Q_f (I + D) J_k.  Where
// theta's rows are graded (NS = OZ_S) it is seven digits, exact down to 2^-31 of
// the largest entry, and nothing is rounded.
// BASIS false: the digits alone, of a sketch with m or (use_n) n rows.
// (zs: digits of Ad per instance)
template <bool BASIS, int NS>
__global__ void __launch_bounds__(256) k_oz_digits_q(const Dims* __restrict__ dims,
                                                     const ProbPtr* __restrict__ ptrs, float2* __restrict__ Qf,
                                                     uint16_t* Ad, size_t zs, int* Es, int mc, int lc, int Kp,
                                                     int use_n, int cond) {
  const int z = blockIdx.y;
  const Dims D = dims[z];
  if (!D.active || !oz_takes(D, cond)) return;
  const int lane = threadIdx.x & 31;
  const int i = blockIdx.x * 8 + (threadIdx.x >> 5);
  if (i >= lc) return;
  const int Mi = use_n ? D.n : D.m, K = i < D.l ? Mi : 0;
  float2* q = Qf + (size_t)z * mc * lc + (size_t)i * mc;
  cplx* Qd = ptrs[z].Q + (size_t)i * D.m;  // (i < D.l where it is written)
  int E = 0;
  for (int k = lane; k < K; k += 32) {
    const float2 v = q[k];
    E = max(E, max(oz_exp(v.x), oz_exp(v.y)));
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) E = max(E, __shfl_xor_sync(0xffffffffu, E, o));
  if (lane == 0) Es[(size_t)z * lc + i] = E;
  // x = N 2^(E - 1023 - 30), the scale as an FP32 number (a Q_f column has unit norm: E far from its ends)
  const float unit = __uint_as_float((unsigned)max(1, min(254, E - 1023 - 30 + 127)) << 23);
  uint16_t* base = Ad + z * zs;
  const int kend = min(Kp, ((Mi + OZ_KB - 1) / OZ_KB) * OZ_KB);
  for (int k = 4 * lane; k < kend; k += 128) {
    int64_t nr[4], ni[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const float2 v = (k + u < K) ? q[k + u] : make_float2(0.f, 0.f);
      nr[u] = oz_fix_f32<NS>(v.x, E);
      ni[u] = oz_fix_f32<NS>(v.y, E);
      if (BASIS && k + u < K) {
        float2 r = v;
        if (NS == OZ_SQ) {
          r = make_float2((float)(int)nr[u] * unit, (float)(int)ni[u] * unit);
          q[k + u] = r;
        }
        Qd[k + u] = cmk((double)r.x, (double)r.y);
      }
    }
    uint2 d[NS];
    uint16_t* at = base + oz_at<NS>(k >> 4, 0, i, (k >> 3) & 1, lc) + (k & 4);
    oz_digits4<NS>(nr, d);
#pragma unroll
    for (int t = 0; t < NS; ++t) *reinterpret_cast<uint2*>(at + (size_t)t * lc * OZ_KS) = d[t];
    oz_digits4<NS>(ni, d);
#pragma unroll
    for (int t = 0; t < NS; ++t) *reinterpret_cast<uint2*>(at + (size_t)(NS + t) * lc * OZ_KS) = d[t];
  }
}

// ---------------------------------------------------------------------------
// The digit-pair GEMM.
// ---------------------------------------------------------------------------
struct OzArgs {
  const uint16_t* Ad;  // digits of both operands (oz_at)
  const uint16_t* Bd;
  int lc, nc, Kp;      // capacities: rows of C, columns of C, padded k
  size_t az, bz;       // digits per instance
  const int* As;       // [z][i] largest biased exponents of the left operand's rows
  const int* Bs;       // [z][j]
  int* err;
  uint32_t poll_limit;
  int stall;
  int cond;            // which problems the launch takes (DPC_*)
};

__device__ __forceinline__ void oz_bulk_load(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                   tc_smem_u32(dst)),
               "l"(src), "r"(bytes), "r"(tc_smem_u32(bar))
               : "memory");
}

// Shared-memory descriptor, K-major, 32-byte swizzle: 8-row atoms of 256
// bytes (stride byte offset 256).  The low word holds the address (in units
// of 16 bytes; the offsets below stay inside its 14 bits) and the leading
// byte offset (unused: one atom along k); the high word is a constant.
enum : uint32_t { OZ_DESC_HI = (256u >> 4) | (1u << 14) | (6u << 29) };  // stride, version, 32-byte swizzle
__device__ __forceinline__ uint32_t oz_desc_lo(uint32_t saddr) { return ((saddr >> 4) & 0x3FFFu) | (1u << 16); }

// kind::f16 instruction descriptor: D = F32, A = B = BF16, K-major, M x N.
__host__ __device__ constexpr uint32_t oz_idesc(int M, int N, bool negA) {
  return (1u << 4) | (1u << 7) | (1u << 10) | (negA ? (1u << 13) : 0u) | ((uint32_t)(N >> 3) << 17) |
         ((uint32_t)(M >> 4) << 24);
}

// One MMA by the lane with leader != 0 (the warp runs the issue loop uniformly:
// descriptors then stay in uniform registers).
__device__ __forceinline__ void oz_mma(uint32_t leader, uint32_t d, uint32_t alo, uint32_t blo, uint32_t idesc,
                                       uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t.reg .b64 a, b;\n\t"
      "setp.ne.b32 p, %5, 0;\n\t"
      "setp.ne.b32 q, %0, 0;\n\t"
      "mov.b64 a, {%2, %6};\n\t"
      "mov.b64 b, {%3, %6};\n\t"
      "@q tcgen05.mma.cta_group::1.kind::f16 [%1], a, b, %4, p;\n\t}\n" ::"r"(leader),
      "r"(d), "r"(alo), "r"(blo), "r"(idesc), "r"(acc), "r"((uint32_t)OZ_DESC_HI)
      : "memory");
}

__device__ __forceinline__ void oz_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(tc_smem_u32(bar))
               : "memory");
}

__device__ __forceinline__ void oz_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(tc_smem_u32(bar)) : "memory");
}

// Warp-uniform bounded wait: lane 0 polls, the warp gets its answer.
__device__ __forceinline__ bool oz_warp_wait(uint64_t* bar, uint32_t parity, uint32_t limit, int* err,
                                             volatile int* abort_flag) {
  bool ok = false;
  if ((threadIdx.x & 31) == 0) ok = tc_mbar_wait(bar, parity, limit, err, abort_flag);
  return __shfl_sync(0xffffffffu, ok ? 1 : 0, 0) != 0;
}

// two consecutive accumulator columns of this warp's 32 lanes
__device__ __forceinline__ void oz_ld2(uint32_t taddr, float* v) {
  uint32_t r0, r1;
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x2.b32 {%0, %1}, [%2];" : "=r"(r0), "=r"(r1) : "r"(taddr) : "memory");
  v[0] = __uint_as_float(r0);
  v[1] = __uint_as_float(r1);
}

// (hi, lo) += the seven level sums v[0], v[1], ... (levels 2 .. 8): hi counts
// units of level 6, lo (FP32) units of level 8.  Levels 2 and 3 (below 2^22)
// become integers by adding 1.5 2^23, the others by conversion.
__device__ __forceinline__ void oz_add_levels(int64_t& hi, float& lo, const float (*v)[2], int q) {
  const float magic = 12582912.f;  // 1.5 2^23: the low bits of the sum are the integer
  const unsigned mb = 0x4B400000u;
  const int i01 = (int)(__float_as_uint(v[0][q] + magic) * 256u + __float_as_uint(v[1][q] + magic) - mb * 257u);
  const int i2 = __float2int_rn(v[2][q]), i3 = __float2int_rn(v[3][q]), i4 = __float2int_rn(v[4][q]);
  hi += (int64_t)i01 * 16777216;
  hi += (int64_t)i2 * 65536;
  hi += (int64_t)i3 * 256;
  hi += i4;
  lo += fmaf(v[5][q], 256.f, v[6][q]);
}

template <int ST>
__global__ void __launch_bounds__(OZ_THREADS, 1)
    k_oz_gemm(const Dims* __restrict__ dims, const ProbPtr* __restrict__ ptrs, OzArgs a) {
  typedef OzGeo<ST> Geo;
  constexpr int SA = Geo::SA, SB = Geo::SB, STAGES = Geo::STAGES;
  extern __shared__ __align__(1024) uint8_t oz_smem_raw[];
  const int z = blockIdx.z;
  const Dims D = dims[z];
  const int i0 = blockIdx.y * OZ_BM, j0 = blockIdx.x * OZ_BN;
  if (!D.active || !oz_takes(D, a.cond) || oz_skip<ST>(D, ptrs[z])) return;
  const OzOp op = oz_op<ST>(D, ptrs[z]);
  if (i0 >= op.M || j0 >= op.N) return;  // uniform: before any barrier or allocation
  uint8_t* smem = (uint8_t*)(((uintptr_t)oz_smem_raw + 1023) & ~(uintptr_t)1023);
  uint8_t* sA = smem;
  uint8_t* sB = smem + STAGES * Geo::A_STAGE;
  uint64_t* full = (uint64_t*)(sB + STAGES * Geo::B_STAGE);
  uint64_t* empty = full + STAGES;
  uint64_t* accf = empty + STAGES;
  uint64_t* accfree = accf + 1;
  uint64_t* drain = accfree + 1;
  uint32_t* tmem_holder = (uint32_t*)(drain + 1);
  volatile int* abort_flag = (volatile int*)(tmem_holder + 1);

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int nks = (min(op.K, a.Kp) + OZ_KS - 1) / OZ_KS;  // k steps of this instance
  const int nkb = (nks + OZ_DRAIN / OZ_KS - 1) / (OZ_DRAIN / OZ_KS);  // exact accumulation blocks

  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(tc_smem_u32(tmem_holder)),
                 "r"((uint32_t)OZ_TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (tid == 32) {
    for (int s = 0; s < STAGES; ++s) {
      tc_mbar_init(&full[s], 1);
      tc_mbar_init(&empty[s], 1);
    }
    tc_mbar_init(accf, 1);
    tc_mbar_init(accfree, OZ_EPI_WARPS);
    tc_mbar_init(drain, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_holder;

  if (warp == 0) {
    // ---- producer: per k step one bulk copy per plane and operand (lanes
    // 0 .. 2 SA - 1 the left operand's, the next 2 SB the right one's); rows past the
    // arrays' own are not copied, and what those rows of the tile hold only
    // reaches outputs that are not stored.
    const bool isA = lane < 2 * SA;
    const int plane = isA ? lane : lane - 2 * SA, row0 = isA ? i0 : j0, rc = isA ? a.lc : a.nc;
    const int na = min((int)OZ_BM, a.lc - i0), nb = min((int)OZ_BN, a.nc - j0);  // rows copied
    const uint32_t bytes = (uint32_t)(isA ? na : nb) * (OZ_KS * 2);
    const uint16_t* src = (isA ? a.Ad : a.Bd) + z * (isA ? a.az : a.bz) + ((size_t)plane * rc + row0) * OZ_KS;
    const size_t step = (size_t)(isA ? 2 * SA : 2 * SB) * rc * OZ_KS;
    uint8_t* dst = (isA ? sA : sB) + (size_t)plane * (isA ? OZ_A_TILE : OZ_B_TILE);
    const uint32_t stage = isA ? Geo::A_STAGE : Geo::B_STAGE;
    int issued = 0;
    bool ok = true;
    for (int it = 0; it < (a.stall ? 0 : nks); ++it) {
      const int s = it % STAGES;
      const uint32_t r = (uint32_t)(it / STAGES);
      if (it >= STAGES && !(ok = oz_warp_wait(&empty[s], (r & 1u) ^ 1u, a.poll_limit, a.err, abort_flag))) break;
      if (lane == 0) tc_mbar_expect_tx(&full[s], (uint32_t)(na * SA + nb * SB) * (2 * OZ_KS * 2));
      __syncwarp();
      if (lane < 2 * (SA + SB)) oz_bulk_load(dst + (size_t)s * stage, src + (size_t)it * step, bytes, &full[s]);
      issued = it + 1;
    }
    if (lane == 0 && *abort_flag) {  // every copy issued lands before the teardown
      for (int it = (issued > STAGES ? issued - STAGES : 0); it < issued; ++it)
        for (uint32_t i = 0; i < (1u << 22); ++i)
          if (tc_mbar_try_wait(&full[it % STAGES], (uint32_t)(it / STAGES) & 1u)) break;
    }
    __syncwarp();
  } else if (warp == 1) {
    // ---- MMA issuer: per k step the digit pairs (t, u) with t + u <= 8, as
    // one MMA per digit t of A and real product; all lanes run the loop, lane
    // 0 issues
    const uint32_t leader = lane == 0 ? 1u : 0u;
    const uint32_t a0 = oz_desc_lo(tc_smem_u32(sA)), b0 = oz_desc_lo(tc_smem_u32(sB));
    bool ok = true;
    int issued_mma = 0, s = 0, it = 0;
    uint32_t ph = 0;
    for (int kb = 0; kb < nkb && ok; ++kb) {
      if (kb > 0 && !(ok = oz_warp_wait(accfree, (uint32_t)(kb - 1) & 1u, a.poll_limit, a.err, abort_flag))) break;
      for (int ks = 0; ks < OZ_DRAIN / OZ_KS && it < nks; ++ks, ++it) {
        if (!(ok = oz_warp_wait(&full[s], ph, a.poll_limit, a.err, abort_flag))) break;
        tc_fence_after();
        const uint32_t as = a0 + (uint32_t)s * (Geo::A_STAGE >> 4), br = b0 + (uint32_t)s * (Geo::B_STAGE >> 4);
        const uint32_t bi = br + SB * (OZ_B_TILE >> 4);
        const uint32_t first = ks == 0 ? 0u : 1u;
        // digit t of A times planes u = 1 .. min(SB, 8 - t) of B (adjacent in
        // shared memory) into the accumulators of levels t + 1 .. (adjacent in
        // tensor memory).  The t = 1 MMAs of a block's first k step start the
        // sums of the levels they cover; with SB < 7 the levels above SB + 1
        // start with the first larger t that reaches them
#pragma unroll
        for (int t = 1; t <= SA; ++t) {
          constexpr bool cA = OzConj<ST>::A;  // a conjugated left operand: C_r = Ar Br + Ai Bi, C_i = Ar Bi - Ai Br
          const int nu = SB < OZ_S + 1 - t ? SB : OZ_S + 1 - t;
          const uint32_t ar = as + (t - 1) * (OZ_A_TILE >> 4), ai = as + (SA + t - 1) * (OZ_A_TILE >> 4);
          const uint32_t dr = tmem + (uint32_t)(OZ_BN * (t - 1)), di = dr + (uint32_t)(OZ_BN * OZ_NGRP);
          // planes 1 .. nu - 1 reach levels earlier digits t have started (t > 1);
          // the last plane of a short right operand opens a new level
          const bool opens = t > 1 && SB < OZ_S + 1 - (t - 1) && nu == SB;
          const int n0 = opens ? nu - 1 : nu;
          const uint32_t acc0 = t == 1 ? first : 1u;
          const uint32_t ip = oz_idesc(OZ_BM, OZ_BN * n0, false), in = oz_idesc(OZ_BM, OZ_BN * n0, true);
          oz_mma(leader, dr, ar, br, ip, acc0);                         // C_r += Ar Br
          oz_mma(leader, dr, ai, bi, cA ? ip : in, 1u);                 // C_r -= Ai Bi
          oz_mma(leader, di, ar, bi, ip, acc0);                         // C_i += Ar Bi
          oz_mma(leader, di, ai, br, cA ? in : ip, 1u);                 // C_i += Ai Br
          if (opens) {
            const uint32_t jp = oz_idesc(OZ_BM, OZ_BN, false), jn = oz_idesc(OZ_BM, OZ_BN, true);
            const uint32_t off = (uint32_t)(OZ_BN * n0), bo = n0 * (OZ_B_TILE >> 4);
            oz_mma(leader, dr + off, ar, br + bo, jp, first);
            oz_mma(leader, dr + off, ai, bi + bo, cA ? jp : jn, 1u);
            oz_mma(leader, di + off, ar, bi + bo, jp, first);
            oz_mma(leader, di + off, ai, br + bo, cA ? jn : jp, 1u);
          }
        }
        if (leader) oz_commit(&empty[s]);  // the stage is free once these MMAs have read it
        issued_mma = 1;
        if (++s == STAGES) {
          s = 0;
          ph ^= 1u;
        }
      }
      if (!ok) break;
      if (leader) oz_commit(accf);  // block kb's sums are ready
    }
    if (!ok && leader) {
      *abort_flag = 1;
      if (issued_mma > 0) {  // the MMAs issued read shared memory and write the tensor memory freed below
        oz_commit(drain);
        for (uint32_t i = 0; i < a.poll_limit; ++i)
          if (tc_mbar_try_wait(drain, 0)) break;
      }
    }
    __syncwarp();
  } else {
    // ---- epilogue: warp w reads lanes 32 (w % 4) .. +31 and a quarter of the columns
    const int ew = warp - 2, quad = warp & 3, part = ew >> 2;
    const int i = i0 + 32 * quad + lane;  // row of C
    const int jq = j0 + 8 * part;         // first column of this warp
    int64_t hr[8], hi[8];  // sums (Re, Im) of 8 columns in units of level 6
    float lr[8], li[8];    // levels 7 and 8, in units of level 8
    volatile double ext[16];  // what OZ_FLUSH blocks moved out of hr, hi (depths above 64 OZ_FLUSH only)
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      hr[c] = hi[c] = 0;
      lr[c] = li[c] = 0.f;
    }
    const bool deep = nkb > OZ_FLUSH;
    if (deep)
      for (int c = 0; c < 16; ++c) ext[c] = 0.0;
    bool ok = true;
    const uint32_t lanes = tmem + ((uint32_t)(32 * quad) << 16) + (uint32_t)(8 * part);
    for (int kb = 0; kb < nkb; ++kb) {
      if (!(ok = oz_warp_wait(accf, (uint32_t)kb & 1u, a.poll_limit, a.err, abort_flag))) break;
      tc_fence_after();
#pragma unroll
      for (int c2 = 0; c2 < 8; c2 += 2) {  // two columns of every accumulator per load
        float v[2 * OZ_NGRP][2];
#pragma unroll
        for (int g = 0; g < 2 * OZ_NGRP; ++g) oz_ld2(lanes + (uint32_t)(OZ_BN * g + c2), v[g]);
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
        if (c2 == 6) {  // everything is in registers: the accumulators may be overwritten
          tc_fence_before();
          __syncwarp();
          if (lane == 0) oz_arrive(accfree);
        }
#pragma unroll
        for (int q = 0; q < 2; ++q) {
          oz_add_levels(hr[c2 + q], lr[c2 + q], v, q);
          oz_add_levels(hi[c2 + q], li[c2 + q], v + OZ_NGRP, q);
        }
      }
      if (deep && (kb % OZ_FLUSH) == OZ_FLUSH - 1) {
#pragma unroll
        for (int c = 0; c < 8; ++c) {
          ext[c] = ext[c] + (double)hr[c];
          ext[8 + c] = ext[8 + c] + (double)hi[c];
          hr[c] = hi[c] = 0;
        }
      }
    }
    if (ok && i < op.M) {
      // (the digits of a short operand are those of N 2^24, its integer in the units of a full one)
      const double sa = oz_scale(a.As[(size_t)z * a.lc + i]);
#pragma unroll
      for (int c = 0; c < 8; ++c) {
        const int j = jq + c;
        if (j < op.N) {
          const double sc = sa * oz_scale(a.Bs[(size_t)z * a.nc + j]);
          double re = fma((double)lr[c], 1.52587890625e-5, (double)hr[c]);  // level 8 = 2^-16 of level 6
          double im = fma((double)li[c], 1.52587890625e-5, (double)hi[c]);
          if (deep) {
            re += ext[c];
            im += ext[8 + c];
          }
          oz_store<ST>(D, ptrs[z], op, i, j, re * sc, im * sc);
        }
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"((uint32_t)OZ_TMEM_COLS)
                 : "memory");
  }
}


// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
int oz_kpad(int m) { return ((m + OZ_KB - 1) / OZ_KB) * OZ_KB; }

size_t oz_digits_bytes(int rows, int m) { return (size_t)2 * OZ_S * rows * oz_kpad(m) * sizeof(uint16_t); }
size_t oz_digits_q_bytes(int rows, int m) { return (size_t)2 * OZ_SQ * rows * oz_kpad(m) * sizeof(uint16_t); }
size_t oz_scales_bytes(int rows) { return (size_t)rows * sizeof(int); }

template <int ST>
static cudaError_t oz_launch(int Mc, int Nc, int batch, const Dims* dims, const ProbPtr* ptrs, const OzArgs& oa,
                             cudaStream_t st) {
  k_oz_gemm<ST><<<dim3((Nc + OZ_BN - 1) / OZ_BN, (Mc + OZ_BM - 1) / OZ_BM, batch), OZ_THREADS, OzGeo<ST>::smem, st>>>(
      dims, ptrs, oa);
  return cudaGetLastError();
}

template <int ST>
static cudaError_t oz_attr() {
  return cudaFuncSetAttribute(k_oz_gemm<ST>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)OzGeo<ST>::smem);
}

cudaError_t oz_prepare() {
  static DeviceOnce once;
  return once([] {
    const cudaError_t es[] = {
        oz_attr<OZ_CONT>(), oz_attr<OZ_GRAMY>(), oz_attr<OZ_GRAMT>(),
        oz_attr<OZ_PROJ7>(), oz_attr<OZ_GRAM7>(),
        oz_attr<OZ_PROJ>(), oz_attr<OZ_GRAM>(), oz_attr<OZ_THETA>(), oz_attr<OZ_GATE>(), oz_attr<G_X>(),
        oz_attr<G_U>(),     oz_attr<G_V>(),     oz_attr<G_Y0>(),     oz_attr<G_Y>(),     oz_attr<G_YT>(),
        oz_attr<G_BH>(),    oz_attr<G_PR>(),    oz_attr<G_PQ>(),     oz_attr<G_PD>(),    oz_attr<G_CYG>(),
        oz_attr<G_CYQ>(),   oz_attr<G_CQG>(),   oz_attr<G_CQQ>(),    oz_attr<G_CTG>(),   oz_attr<G_CTQ>(),
        oz_attr<G_CRG>(),   oz_attr<G_CRQ>(),   oz_attr<G_JG>(),     oz_attr<G_JT>(),    oz_attr<G_XJ>(),
        oz_attr<G_XG>(),    oz_attr<G_XT>()};
    for (cudaError_t e : es)
      if (e != cudaSuccess) return e;
    return cudaSuccess;
  });
}

// Capacities (rows of C, columns of C, depth) of a stage's product.
static void oz_stage_caps(int stage, const Caps& c, int& Mc, int& Nc, int& Kc) {
  switch (stage) {
    case G_Y0: case G_Y: Mc = c.m; Nc = c.l; Kc = c.n; break;
    case G_YT: case G_BH: Mc = c.n; Nc = c.l; Kc = c.m; break;
    case G_PR: Mc = c.m; Nc = c.r; Kc = c.n; break;
    case G_PQ: Mc = c.l; Nc = c.r; Kc = c.m; break;
    case G_PD: Mc = c.m; Nc = c.r; Kc = c.l; break;
    case G_CYG: case G_CQG: Mc = c.l; Nc = c.l; Kc = c.m; break;
    case G_CYQ: case G_CQQ: Mc = c.m; Nc = c.l; Kc = c.l; break;
    case G_CTG: case G_CRG: case G_X: Mc = c.l; Nc = c.l; Kc = c.n; break;
    case G_CTQ: case G_CRQ: Mc = c.n; Nc = c.l; Kc = c.l; break;
    case G_JG: case G_JT: case G_XJ: case G_XG: case G_XT: Mc = c.l; Nc = c.l; Kc = c.l; break;
    case G_U: Mc = c.m; Nc = c.k; Kc = c.l; break;
    case OZ_THETA: case OZ_CONT: Mc = c.m; Nc = c.n; Kc = c.cm; break;  // K = chi_m, at most its bond's capacity
    case OZ_GATE: Mc = c.dl * c.dr; Nc = c.cl * c.cr; Kc = c.dl * c.dr; break;
    default: Mc = c.n; Nc = c.k; Kc = c.l; break;  // G_V
  }
}

bool oz_stage_rule(const Caps& cap) { return cap.l >= 48 && (cap.m >= 256 || cap.n >= 256); }

static const int OZ_STAGE_LIST[] = {G_CTG, G_CTQ, G_X, G_U, G_V};

static void oz_grow(OzStageBytes& b, int stage, const Caps& c) {
  int Mc, Nc, Kc;
  oz_stage_caps(stage, c, Mc, Nc, Kc);
  b.ad = std::max(b.ad, oz_digits_bytes(Mc, Kc));
  b.as = std::max(b.as, oz_scales_bytes(Mc));
  b.bd = std::max(b.bd, oz_digits_bytes(Nc, Kc));
  b.bs = std::max(b.bs, oz_scales_bytes(Nc));
}

OzStageBytes oz_stage_bytes(int m, int n, int k, int l, const Caps* gate) {
  OzStageBytes b{0, 0, 0, 0};
  Caps c{};
  c.m = m; c.n = n; c.k = k; c.l = l;
  for (int stage : OZ_STAGE_LIST) oz_grow(b, stage, c);
  b.ad = std::max(b.ad, oz_digits_q_bytes(l, std::max(m, n)));  // of the FP32 sketches
  if (gate && theta_digits_rule(gate->m, gate->n, gate->cm)) oz_grow(b, OZ_CONT, *gate);
  if (gate && gate->dl * gate->dr >= GATE_GEMM_MIN) {
    oz_grow(b, OZ_THETA, *gate);
    oz_grow(b, OZ_GATE, *gate);
  }
  return b;
}

bool oz_gate_rule(const Caps& cap) { return cap.dl * cap.dr >= GATE_GEMM_MIN; }

// Digits and exponents of one operand (rows rc, padded depth Kp).
template <int ST, int SIDE>
static cudaError_t oz_digits(const Dims* dims, const ProbPtr* ptrs, int batch, int rc, int Kp, uint16_t* Xd, int* Es,
                             int cond, cudaStream_t st, const char* label = "k_oz_digits[op]") {
  ProfScope ps(label, st);
  if (Kp <= OZ_SELF_K) {
    k_oz_digits_op<ST, SIDE, true><<<dim3((rc + 15) / 16, 1, batch), 256, 0, st>>>(dims, ptrs, Xd, Es, rc, Kp, cond);
  } else {
    const cudaError_t e = cudaMemsetAsync(Es, 0, sizeof(int) * (size_t)rc * batch, st);
    if (e != cudaSuccess) return e;
    k_oz_max<ST, SIDE><<<dim3((rc + 15) / 16, (Kp + OZ_MAX_K - 1) / OZ_MAX_K, batch), 256, 0, st>>>(dims, ptrs, Es,
                                                                                                   rc, cond);
    k_oz_digits_op<ST, SIDE, false><<<dim3((rc + 15) / 16, Kp / OZ_KB, batch), 256, 0, st>>>(dims, ptrs, Xd, Es, rc,
                                                                                             Kp, cond);
  }
  return cudaGetLastError();
}

// One product; pre: the left operand's digits where they are already made
// (theta's), else they go to the scratch.
template <int ST>
static cudaError_t oz_stage_run(const Dims* dims, const ProbPtr* ptrs, int batch, int Mc, int Nc, int Kc,
                                const OzScratch& sc, int cond, int* err, cudaStream_t st,
                                const uint16_t* pre = nullptr, const int* pre_es = nullptr) {
  const int Kp = oz_kpad(Kc);
  // an operand times its own adjoint: one set of digits
  constexpr bool same = ST == G_CYG || ST == G_CQG || ST == G_CTG || ST == G_CRG ||
                        ST == G_JG || ST == G_XG;
  cudaError_t e = cudaSuccess;
  if constexpr (ST == OZ_THETA || ST == OZ_CONT) {
    ProfScope ps("k_oz_balance", st);
    k_oz_balance<ST><<<dim3((Kc + 31) / 32, batch), 256, 0, st>>>(dims, ptrs, cond);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  if (!same && !pre && Kp <= OZ_SELF_K) {
    if constexpr (!same) {
      ProfScope ps("k_oz_digits[op]", st);
      k_oz_digits_two<ST><<<dim3((std::max(Mc, Nc) + 15) / 16, 2, batch), 256, 0, st>>>(dims, ptrs, sc.ad, sc.as, Mc,
                                                                                        sc.bd, sc.bs, Nc, Kp, cond);
      e = cudaGetLastError();
    }
  } else {
    if (!pre) e = oz_digits<ST, 0>(dims, ptrs, batch, Mc, Kp, sc.ad, sc.as, cond, st);
    if constexpr (!same)
      if (e == cudaSuccess) e = oz_digits<ST, 1>(dims, ptrs, batch, Nc, Kp, sc.bd, sc.bs, cond, st);
  }
  if (e != cudaSuccess) return e;
  const uint16_t* ad = pre ? pre : sc.ad;
  OzArgs oa;
  oa.Ad = ad;
  oa.Bd = same ? ad : sc.bd;
  oa.lc = Mc;
  oa.nc = Nc;
  oa.Kp = Kp;
  oa.az = (size_t)2 * OZ_S * Mc * Kp;
  oa.bz = (size_t)2 * OZ_S * Nc * Kp;
  oa.As = pre ? pre_es : sc.as;
  oa.Bs = same ? oa.As : sc.bs;
  oa.err = err;
  oa.poll_limit = 1u << 24;
  oa.stall = 0;
  oa.cond = cond;
  ProfScope ps(ST == G_U || ST == G_V ? "k_oz_gemm[uv]"
               : ST == OZ_THETA || ST == OZ_CONT ? "k_oz_gemm[theta]"
               : ST == OZ_GATE           ? "k_oz_gemm[gate]"
               : ST >= G_JG && ST <= G_XT ? "k_oz_gemm[svd]"
               : ST <= G_BH || (ST >= G_PR && ST <= G_PD) ? "k_oz_gemm[sketch]"
                                         : "k_oz_gemm[cholqr]",
               st);
  return oz_launch<ST>(Mc, Nc, batch, dims, ptrs, oa, st);
}

cudaError_t launch_oz_stage(int stage, const Dims* dims, const ProbPtr* ptrs, int batch, const Caps& cap,
                            const OzScratch& sc, int* err, cudaStream_t st, int cond) {
  const cudaError_t e = oz_prepare();
  if (e != cudaSuccess) return e;
  int Mc, Nc, Kc;
  oz_stage_caps(stage, cap, Mc, Nc, Kc);
#define OZ_CASE(S) \
  case S: return oz_stage_run<S>(dims, ptrs, batch, Mc, Nc, Kc, sc, cond, err, st)
  switch (stage) {
    case OZ_THETA:
    case OZ_GATE:
      if (!oz_gate_rule(cap)) return cudaSuccess;
      return stage == OZ_THETA ? oz_stage_run<OZ_THETA>(dims, ptrs, batch, Mc, Nc, Kc, sc, cond, err, st)
                               : oz_stage_run<OZ_GATE>(dims, ptrs, batch, Mc, Nc, Kc, sc, cond, err, st);
    OZ_CASE(OZ_CONT);
    OZ_CASE(G_X);
    OZ_CASE(G_U);
    OZ_CASE(G_V);
    OZ_CASE(G_PQ);
    OZ_CASE(G_PD);
    OZ_CASE(G_CYG);
    OZ_CASE(G_CYQ);
    OZ_CASE(G_CQG);
    OZ_CASE(G_CQQ);
    OZ_CASE(G_CTG);
    OZ_CASE(G_CTQ);
    OZ_CASE(G_CRG);
    OZ_CASE(G_CRQ);
    OZ_CASE(G_JG);
    OZ_CASE(G_JT);
    OZ_CASE(G_XJ);
    OZ_CASE(G_XG);
    OZ_CASE(G_XT);
    default: return cudaErrorInvalidValue;
  }
#undef OZ_CASE
}

// The same for a batch in runs of `chunk` problems, which share the scratch.
cudaError_t launch_oz_range(int stage, const Dims* dims, const ProbPtr* ptrs, int batch, const Caps& cap,
                            const OzScratch& sc, int chunk, int cond, int* err, cudaStream_t st) {
  for (int z = 0; z < batch; z += chunk) {
    const cudaError_t e = launch_oz_stage(stage, dims + z, ptrs + z, std::min(chunk, batch - z), cap, sc, err, st, cond);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

// ---------------------------------------------------------------------------
// The FP64 form's products with theta.
// ---------------------------------------------------------------------------
struct DpLayout {
  size_t tr, tc, er, ec, ad, as, bd, bs;  // bytes per problem
  size_t per(bool both) const { return (both ? tr + tc : std::max(tr, tc)) + er + ec + ad + as + bd + bs; }
};

static DpLayout dp_layout(const Caps& c) {
  DpLayout d;
  const int mx = std::max(c.m, c.n), w = std::max(c.l, std::max(c.k, c.r));
  d.tr = oz_digits_bytes(c.m, c.n);
  d.tc = oz_digits_bytes(c.n, c.m);
  d.er = oz_scales_bytes(c.m);
  d.ec = oz_scales_bytes(c.n);
  // left operands: l or mx rows, depths mx or l; right ones: w rows
  d.ad = std::max(oz_digits_bytes(c.l, mx), oz_digits_bytes(mx, c.l));
  d.as = oz_scales_bytes(std::max(mx, c.l));
  d.bd = std::max(oz_digits_bytes(w, mx), oz_digits_bytes(w, c.l));
  d.bs = oz_scales_bytes(w);
  if (theta_digits_rule(c.m, c.n, c.cm)) {  // a handle's contraction
    d.ad = std::max(d.ad, oz_digits_bytes(c.m, c.cm));
    d.bd = std::max(d.bd, oz_digits_bytes(c.n, c.cm));
    d.bs = std::max(d.bs, oz_scales_bytes(c.n));
  }
  return d;
}

static size_t dp_up(size_t x) { return (x + 255) & ~(size_t)255; }

static int dp_chunk(const DpLayout& d, int batch, size_t limit, int* all) {
  *all = d.per(true) * batch <= limit;
  if (*all) return batch;
  const size_t c = limit / d.per(false);
  return c < 1 ? 1 : (c < (size_t)batch ? (int)c : batch);
}

size_t dp_bytes(const Caps& cap, int batch, size_t limit) {
  const DpLayout d = dp_layout(cap);
  int all;
  const size_t c = dp_chunk(d, batch, limit, &all);
  return (all ? dp_up(d.tr * c) + dp_up(d.tc * c) : dp_up(std::max(d.tr, d.tc) * c)) + dp_up(d.er * c) +
         dp_up(d.ec * c) + dp_up(d.ad * c) + dp_up(d.as * c) + dp_up(d.bd * c) + dp_up(d.bs * c);
}

DpScratch dp_carve(char* base, const Caps& cap, int batch, size_t limit, int* err) {
  const DpLayout d = dp_layout(cap);
  DpScratch s;
  s.chunk = dp_chunk(d, batch, limit, &s.all);
  s.err = err;
  const size_t c = s.chunk;
  size_t o = 0;
  auto take = [&](size_t bytes) {
    char* q = base + o;
    o += dp_up(bytes * c);
    return q;
  };
  if (s.all) {
    s.tr = (uint16_t*)take(d.tr);
    s.tc = (uint16_t*)take(d.tc);
  } else {
    s.tr = s.tc = (uint16_t*)take(std::max(d.tr, d.tc));
  }
  s.er = (int*)take(d.er);
  s.ec = (int*)take(d.ec);
  s.oz.ad = (uint16_t*)take(d.ad);
  s.oz.as = (int*)take(d.as);
  s.oz.bd = (uint16_t*)take(d.bd);
  s.oz.bs = (int*)take(d.bs);
  return s;
}

// theta's digits: rows (for Y = A X) or columns (for A^H Q)
static cudaError_t dp_theta(const DpPath& p, int z, int cnt, bool rows) {
  return rows ? oz_digits<G_Y, 0>(p.dims + z, p.ptrs + z, cnt, p.cap.m, oz_kpad(p.cap.n), p.dp->tr, p.dp->er, DPC_DIG,
                                  p.st, "k_oz_digits[theta]")
              : oz_digits<G_YT, 0>(p.dims + z, p.ptrs + z, cnt, p.cap.n, oz_kpad(p.cap.m), p.dp->tc, p.dp->ec, DPC_DIG,
                                   p.st, "k_oz_digits[theta]");
}

cudaError_t dp_begin(const DpPath& p) {
  if (!p.dp || !p.dp->all) return cudaSuccess;
  cudaError_t e = dp_theta(p, 0, p.batch, true);
  return e == cudaSuccess ? dp_theta(p, 0, p.batch, false) : e;
}

cudaError_t launch_dp_stage(int stage, const DpPath& p, int cond) {
  const DpScratch& s = *p.dp;
  if (stage != G_Y0 && stage != G_Y && stage != G_YT && stage != G_BH && stage != G_PR)
    return launch_oz_range(stage, p.dims, p.ptrs, p.batch, p.cap, s.oz, s.chunk, cond, s.err, p.st);
  cudaError_t e = oz_prepare();
  if (e != cudaSuccess) return e;
  const bool rows = stage != G_YT && stage != G_BH;
  int Mc, Nc, Kc;
  oz_stage_caps(stage, p.cap, Mc, Nc, Kc);
  for (int z = 0; z < p.batch; z += s.chunk) {
    const int cnt = std::min(s.chunk, p.batch - z);
    if (!s.all && (e = dp_theta(p, z, cnt, rows)) != cudaSuccess) return e;
    const uint16_t* pre = rows ? s.tr : s.tc;
    const int* es = rows ? s.er : s.ec;
    const Dims* dm = p.dims + z;
    const ProbPtr* pp = p.ptrs + z;
    switch (stage) {
      case G_Y0: e = oz_stage_run<G_Y0>(dm, pp, cnt, Mc, Nc, Kc, s.oz, cond, s.err, p.st, pre, es); break;
      case G_Y: e = oz_stage_run<G_Y>(dm, pp, cnt, Mc, Nc, Kc, s.oz, cond, s.err, p.st, pre, es); break;
      case G_PR: e = oz_stage_run<G_PR>(dm, pp, cnt, Mc, Nc, Kc, s.oz, cond, s.err, p.st, pre, es); break;
      case G_YT: e = oz_stage_run<G_YT>(dm, pp, cnt, Mc, Nc, Kc, s.oz, cond, s.err, p.st, pre, es); break;
      default: e = oz_stage_run<G_BH>(dm, pp, cnt, Mc, Nc, Kc, s.oz, cond, s.err, p.st, pre, es); break;
    }
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

cudaError_t DpPath::gemm(int stage) const {
  const int tile = (tiles && stage <= G_V) ? tiles[stage] : 0;
  if (dp) {
    const int chk = (stage >= G_PR && stage <= G_PD) ? DPC_CHK : 0;
    const cudaError_t e = launch_dp_stage(stage, *this, DPC_DIG | chk);
    if (e != cudaSuccess) return e;
    if (dp_rule(cap.m, cap.n, cap.l) && cap.cm == 0) return cudaSuccess;  // a plan: every problem has the same sizes
  }
  return launch_zgemm_tile(stage, tile, dims, ptrs, batch, cap, st);
}

cudaError_t launch_oz_digits_theta(const Dims* dims, const ProbPtr* ptrs, uint16_t* Bd, int* Bs, int m, int n,
                                   int batch, cudaStream_t st) {
  // the columns' exponents are in Bs (k_conv_theta)
  ProfScope ps("k_oz_digits[theta]", st);
  const int Kp = oz_kpad(m);
  k_oz_digits_op<OZ_PROJ, 1, false><<<dim3((n + 15) / 16, Kp / OZ_KB, batch), 256, 0, st>>>(dims, ptrs, Bd, Bs, n, Kp,
                                                                                            0);
  return cudaGetLastError();
}

// The digits of Q_f: per instance four or seven of the seven planes' room.
cudaError_t launch_oz_digits_qf(const Dims* dims, const ProbPtr* ptrs, float2* Qf, uint16_t* Ad, int* As, int m, int l, int batch,
                                cudaStream_t st) {
  const int Kp = oz_kpad(m);
  const size_t zs = (size_t)2 * OZ_S * l * Kp;
  const dim3 grid((l + 7) / 8, batch);
  ProfScope ps("k_oz_digits[q]", st);
  k_oz_digits_q<true, OZ_SQ><<<grid, 256, 0, st>>>(dims, ptrs, Qf, Ad, zs, As, m, l, Kp, 0, DPC_FLAT);
  k_oz_digits_q<true, OZ_S><<<grid, 256, 0, st>>>(dims, ptrs, Qf, Ad, zs, As, m, l, Kp, 0, DPC_GRADED);
  return cudaGetLastError();
}

cudaError_t launch_oz_gram(const Dims* dims, const ProbPtr* ptrs, const uint16_t* Ad, const int* As, int m, int l,
                           int batch, int* err, cudaStream_t st) {
  cudaError_t e = oz_prepare();
  if (e != cudaSuccess) return e;
  const int Kp = oz_kpad(m);
  OzArgs oa;
  oa.Ad = oa.Bd = Ad;
  oa.lc = l;
  oa.nc = l;
  oa.Kp = Kp;
  oa.az = oa.bz = (size_t)2 * OZ_S * l * Kp;
  oa.As = As;
  oa.Bs = As;
  oa.err = err;
  oa.poll_limit = 1u << 24;
  oa.stall = 0;
  oa.cond = DPC_FLAT;
  ProfScope ps("k_oz_gemm[gram]", st);
  if ((e = oz_launch<OZ_GRAM>(l, l, batch, dims, ptrs, oa, st)) != cudaSuccess) return e;
  oa.cond = DPC_GRADED;
  return oz_launch<OZ_GRAM7>(l, l, batch, dims, ptrs, oa, st);
}

cudaError_t launch_oz_gram_f32(const Dims* dims, const ProbPtr* ptrs, const float2* X, uint16_t* Ad, int* As, int M,
                               int l, int use_n, int batch, int cond, int* err, cudaStream_t st) {
  const cudaError_t e = oz_prepare();
  if (e != cudaSuccess) return e;
  const int Kp = oz_kpad(M);
  {
    ProfScope ps("k_oz_digits[q]", st);
    k_oz_digits_q<false, OZ_SQ><<<dim3((l + 7) / 8, batch), 256, 0, st>>>(
        dims, ptrs, const_cast<float2*>(X), Ad, (size_t)2 * OZ_SQ * l * Kp, As, M, l, Kp, use_n, cond);
    const cudaError_t e2 = cudaGetLastError();
    if (e2 != cudaSuccess) return e2;
  }
  OzArgs oa;
  oa.Ad = oa.Bd = Ad;
  oa.lc = oa.nc = l;
  oa.Kp = Kp;
  oa.az = oa.bz = (size_t)2 * OZ_SQ * l * Kp;
  oa.As = oa.Bs = As;
  oa.err = err;
  oa.poll_limit = 1u << 24;
  oa.stall = 0;
  oa.cond = cond;
  ProfScope ps("k_oz_gemm[gram]", st);
  return use_n ? oz_launch<OZ_GRAMT>(l, l, batch, dims, ptrs, oa, st) : oz_launch<OZ_GRAMY>(l, l, batch, dims, ptrs, oa, st);
}

cudaError_t launch_proj_oz(const Dims* dims, const ProbPtr* ptrs, const uint16_t* Ad, const int* As, const uint16_t* Bd, const int* Bs, int m, int n, int l, int batch,
                           int* err, cudaStream_t st) {
  const int Kp = oz_kpad(m);
  {
    cudaError_t e = oz_prepare();
    if (e != cudaSuccess) return e;
    OzArgs oa;
    oa.Ad = Ad;
    oa.Bd = Bd;
    oa.lc = l;
    oa.nc = n;
    oa.Kp = Kp;
    oa.az = (size_t)2 * OZ_S * l * Kp;
    oa.bz = (size_t)2 * OZ_S * n * Kp;
    oa.As = As;
    oa.Bs = Bs;
    oa.err = err;
    // an injected pipeline stall (test hook), never inside a stream capture
    cudaStreamCaptureStatus cap_st = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(st, &cap_st) != cudaSuccess) cap_st = cudaStreamCaptureStatusActive;
    const bool stall = cap_st == cudaStreamCaptureStatusNone && fault_take(TEBD_FAULT_TC_STALL);
    oa.poll_limit = stall ? (1u << 12) : (1u << 24);
    oa.stall = stall ? 1 : 0;
    oa.cond = DPC_FLAT;
    ProfScope ps("k_oz_proj[project]", st);
    if ((e = oz_launch<OZ_PROJ>(l, n, batch, dims, ptrs, oa, st)) != cudaSuccess) return e;
    oa.cond = DPC_GRADED;
    return oz_launch<OZ_PROJ7>(l, n, batch, dims, ptrs, oa, st);
  }
}

}  // namespace tg
