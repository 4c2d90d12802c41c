// Buffers and entry of the mixed-precision RRSVD (mixed.cu).
#pragma once
#include <cuda_runtime.h>
#include <stddef.h>

#include "internal.cuh"

namespace tg {

// Padded sizes of the real-embedded operands of one instance.
struct MixedSizes {
  int bf16;      // 1: the products before the refinement round in BF16 (TEBD_PREC_BF16)
  int K1;        // 2n rounded up to 32: row length of theta's forward copy and of Bt for A X
  int K2;        // 2m rounded up to 32: row length of the adjoint copy and of Bt for A^H X
  int K1b, K2b;  // the same rounded up to 64 for the BF16 copies (128-byte rows)
  int Np;        // 2l rounded up to 16: rows of Bt (tensor-core N)
  int BN;        // tensor-core tile width, min(Np, 256)
  size_t thf, tha, bt, yf, ytf, df;  // bytes per instance
  size_t bd, bsc, ad, asc;  // BF16 digits and row exponents of theta and of Q_f^H (tensor-core projection)
  size_t span;              // exponent range of the last sketch's rows (k_row_span)
  size_t thfb, thab, btb;   // BF16 copies of theta, theta^H and Bt (bf16 only)
  size_t gad, gas, gbd, gbs;  // digit scratch of the other tensor-core products (oz_stage_bytes)
  size_t qs;     // bytes per instance of the many-CTA FP32 QR's scratch (0: not used)
  int ntile;     // 32 x 32 tiles of the theta conversion (partials of ||theta||_F^2)
};

// Batch-major arrays (instance z at base + z * per-instance size).
struct MixedPtrs {
  float* thf_hi;  // m x K1, TF32-rounded theta (Re, Im interleaved)
  float* thf_lo;  // TF32 remainder of theta
  float* tha_hi;  // n x K2, TF32-rounded theta^H
  float* tha_lo;
  float* bt_hi;   // Np x K (K1 or K2), real embedding of the right operand
  float* bt_lo;
  float2* Yf;     // m x l complex FP32, column-major
  float2* Qf;
  float2* Ytf;    // n x l
  float2* Qtf;
  float2* Df;     // l x l correction of the re-orthonormalisation
  uint16_t* bd;   // digits of theta for the tensor-core projection (oz_proj.cu)
  int* bsc;       // their rows' largest exponents
  uint16_t* ad;   // digits of Q_f^H
  int* asc;
  int2* span;
  uint16_t* thf_b;  // m x K1b BF16 theta (bf16 form), or null
  uint16_t* tha_b;  // n x K2b BF16 theta^H
  uint16_t* bt_b;   // Np x max(K1b, K2b) BF16 right operand
  uint16_t* gad;  // digit scratch of the Cholesky QR and U / V products (OzScratch)
  int* gas;
  uint16_t* gbd;
  int* gbs;
  double* tpart;  // ntile partial sums of |theta|^2 per instance
  float2* qscr;   // scratch of the many-CTA FP32 QR (qs bytes per instance), or null
};

MixedSizes mixed_sizes(int m, int n, int k, int l, int bf16 = 0, const Caps* gate = nullptr);
// The arrays of instances z0, z0 + 1, ... of a carve (every array advanced
// by z0 instances): run_rrsvd_mixed on a sub-batch starting at instance z0.
MixedPtrs mixed_offset(const MixedPtrs& p, const MixedSizes& s, int z0);
size_t mixed_bytes(const MixedSizes& s, int batch);
MixedPtrs mixed_carve(char* base, const MixedSizes& s, int batch);

// Blocked FP32 Householder QR (qr_blocked.cu): A (M x L column-major per
// instance, overwritten) -> Q; usable when qr_blk_f32_fits(M, L).  With
// dims, each instance factors only its own rows (D.n if use_n, else D.m) and
// D.l columns of the zero-padded M x L layout.
bool qr_blk_f32_fits(int M, int L);
// threads: 0 picks the CTA size by batch; 128, 256 or 512 force it (when its
// shared memory fits).  rest: only the instances the Cholesky QR gave up (cf)
cudaError_t launch_qr_blk_f32(float2* A, float2* Q, int M, int L, int batch, cudaStream_t st,
                              const Dims* dims = nullptr, int use_n = 0, int threads = 0, int rest = 0);
// The same QR spread over many CTAs per instance (qr_multi.cu), for matrices
// too tall for the blocked kernel's shared memory; scr holds
// qr_multi_f32_scratch(M, L) float2 per instance at the given stride; with
// dims each instance is factored at its own size, as above.
bool qr_multi_f32_fits(int M, int L);
size_t qr_multi_f32_scratch(int M, int L);
cudaError_t launch_qr_multi_f32(float2* A, float2* Q, float2* scr, size_t stride, int M, int L, int batch,
                                cudaStream_t st, const Dims* dims = nullptr, int use_n = 0, int rest = 0);
// The correction D of the re-orthonormalisation Q = Q_f (I + D) (FP64
// orthonormal to ~1e-13, spanning range(Q_f)) from E = Q_f^H Q_f - I already in
// ptrs[z].R (launch_oz_gram); with fold, Q itself into ptrs[z].Q; usable when
// reorth_fits(M, L).
bool reorth_fits(int M, int L);
cudaError_t launch_reorth(const float2* Qf, float2* Dbuf, const Dims* dims, const ProbPtr* ptrs, int M, int L,
                          int batch, int* status, cudaStream_t st, bool fold);
// X <- (I + D) X on the l x l matrix ptrs[z].R (jk = 0: Rb^H of B^H = A^H Q_f
// (I + D) from that of A^H Q_f) or the l x k ptrs[z].Jk (jk = 1: the left
// factors of U = Q_f (I + D) J_k).
cudaError_t launch_fold_small(const float2* Dbuf, const Dims* dims, const ProbPtr* ptrs, int l, int k, int batch,
                              int jk, cudaStream_t st);

// A^H Q_f into ptrs[z].Yt on the tensor cores from BF16 digits (oz_proj.cu):
// launch_oz_digits_theta once theta is in place, launch_oz_digits_qf, then
// launch_proj_oz.  Arrays at capacities m x n (theta) and m x l (Q_f).
int oz_kpad(int m);
size_t oz_digits_bytes(int rows, int m);
size_t oz_digits_q_bytes(int rows, int m);  // of the FP32 basis (four digits)
size_t oz_scales_bytes(int rows);
cudaError_t oz_prepare();
// The other FP64-accurate products on the tensor cores (GemmStage G_G1 ..
// G_X of the Cholesky QR, G_U, G_V): digit scratch of both operands, sized
// by oz_stage_bytes for the capacities, reused by every stage.
struct OzScratch {
  uint16_t* ad;
  int* as;
  uint16_t* bd;
  int* bs;
};
struct OzStageBytes {
  size_t ad, as, bd, bs;  // per instance
};
// gate: the capacities of a TEBD wave whose bonds take the contraction and
// gate GEMMs (stages OZ_THETA, OZ_GATE of launch_oz_stage), or null
OzStageBytes oz_stage_bytes(int m, int n, int k, int l, const Caps* gate = nullptr);
// the contraction and gate GEMMs of a wave on the tensor cores: stages
// OZ_THETA (into the pre-gate buffers) and OZ_GATE (into theta) of
// launch_oz_stage; the wave's bonds without a pre-gate buffer are skipped
enum { OZ_THETA_STAGE = 102, OZ_GATE_STAGE = 103, OZ_CONT_STAGE = 106 };
bool oz_gate_rule(const Caps& cap);
cudaError_t launch_oz_stage(int stage, const Dims* dims, const ProbPtr* ptrs, int batch, const Caps& cap,
                            const OzScratch& sc, int* err, cudaStream_t st, int cond = 0);
// the size rule of MixedKnobs::dfg: the tensor-core products for bonds whose
// products are deep and wide enough to fill the digit-pair pipeline
bool oz_stage_rule(const Caps& cap);

// --- the FP64 form on the tensor cores -------------------------------------
// Scratch of its digit-split products: theta's digits in both directions
// (tr: its rows, tc: its columns) and those of the other operands, for
// `chunk` problems at a time.  all: every problem of the batch has its theta
// digits (made once per truncation); otherwise tr and tc are one buffer,
// filled before each product for a chunk of problems.
struct DpScratch {
  OzScratch oz;
  uint16_t *tr, *tc;
  int *er, *ec;
  int chunk, all;
  int* err;  // tensor-core wait timeout flag
};
// Bytes for `batch` problems of capacities cap, at most `limit` or what one problem needs.
size_t dp_bytes(const Caps& cap, int batch, size_t limit);
DpScratch dp_carve(char* base, const Caps& cap, int batch, size_t limit, int* err);
enum : size_t { DP_LIMIT = (size_t)6 << 30 };  // the FP64 form's scratch: enough to fill the GPU with large problems

// Which QR of Alg. 1 a launch is: the first (of A Omega, as ill-conditioned as
// A), a middle one, the last before the projection (or of B^H), or the first
// when it is the last too.
// (FIRST_LD, CHECK: the bases of the accuracy check, orthonormal to FP64)
enum { DPQ_FIRST = 0, DPQ_MID = 1, DPQ_LAST = 2, DPQ_LAST0 = 3, DPQ_CHECK = 4, DPQ_FIRST_LD = 5 };

// One truncation's launches: products and QRs on whichever path takes each problem.
struct DpPath {
  const Dims* dims;
  const ProbPtr* ptrs;
  int batch;
  const Caps& cap;
  const DpScratch* dp;
  cudaStream_t st;
  const int* tiles;
  cudaError_t gemm(int stage) const;
  cudaError_t qr(int stage, int kind) const;
  cudaError_t svd() const;  // run_jac_pre where it applies; a Jacobi kernel follows
};
cudaError_t dp_begin(const DpPath& p);  // theta's digits, when they are kept
// one digit-split product of the problems selected by cond: bits, and from
// bit 8 up the pass of a Cholesky QR (the problems that take part in it)
// (DPC_WIDE: those of at least DP_WIDE_L columns; a handle's wave also holds bonds
// far below its capacities, whose Householder QR and double-float Jacobi are
// cheaper than the passes and products of the digit forms)
// (DPC_GRADED, DPC_FLAT: by Dims::gr)
enum { DPC_OK = 1, DPC_QFLAG = 2, DPC_DIG = 4, DPC_CHK = 8, DPC_JS = 16, DPC_WIDE = 32, DPC_GRADED = 64, DPC_FLAT = 128,
       DPC_PASS = 8 };
enum { DP_WIDE_L = 40 };
cudaError_t launch_dp_stage(int stage, const DpPath& p, int cond);
// Cholesky QR of Y into Q (side 0) or Yt into Qt (side 1) (cholqr.cu): up to
// `passes` passes, then, with lowdin, the symmetric orthonormalisation to
// FP64 (CQ_PHASES: with the column phases of the Householder QR; CQ_SHIFTED:
// without it, further passes only for the problems a pass shifted);
// min_pivot: the smallest pivot of the scaled Gram matrix accepted in a first
// pass (0: any, by shifted passes).  Problems given up have cf set.
enum { CQ_LOWDIN = 1, CQ_PHASES = 2, CQ_SHIFTED = 4 };
cudaError_t run_cholqr(int side, int passes, int lowdin, float min_pivot, Dims* dims, const ProbPtr* ptrs, int batch,
                       const Caps& cap, const OzScratch& oz, int chunk, int cond, int* err, cudaStream_t st);
// Cholesky QR of an FP32 sketch A (M x l capacities, m or, with use_n, n rows
// per instance) into Q (cholqr.cu): Gram matrices from the digits of A, the
// product in FP32.  last: the basis the FP64 re-orthonormalisation takes.
// Instances given up have cf set (and A as it was).
cudaError_t run_cholqr_f32(float2* A, float2* Q, int M, int l, int use_n, bool last, Dims* dims, const ProbPtr* ptrs,
                           int batch, const OzScratch& oz, int* err, cudaStream_t st);
// Q = A S R^-1 (S R^-1 in FP32 in ptrs[z].J) of the instances of a pass
cudaError_t launch_trmm_f32(const float2* src, float2* dst, const Dims* dims, const ProbPtr* ptrs, int Mc, int Lc,
                            int use_n, int pass, int batch, cudaStream_t st);
// Gram matrix of an FP32 sketch into ptrs[z].R, its digits in Ad / As
cudaError_t launch_oz_gram_f32(const Dims* dims, const ProbPtr* ptrs, const float2* X, uint16_t* Ad, int* As, int M,
                               int l, int use_n, int batch, int cond, int* err, cudaStream_t st);
// The small SVD X J = W S (X in R) of the problems selected by cond, up to the
// tolerance of the Jacobi kernels (Dims::js says how far; jacobi_pre.cu), for
// capacities of jac_pre_rule (whole: the products' scratch holds the whole batch).  fp64: the FP64 kernels' tolerance, else the
// double-float one's.
bool jac_pre_rule(const Caps& cap, bool whole);
cudaError_t jac_pre_prepare();
cudaError_t run_jac_pre(Dims* dims, const ProbPtr* ptrs, int batch, const Caps& cap, const OzScratch& oz, int chunk,
                        int cond, bool fp64, int* err, cudaStream_t st);
cudaError_t launch_jac_none(Dims* dims, int batch, cudaStream_t st);  // js = 0
// T = (J^H J)^-1/2 in Yt from J^H J in Y; js = 0 where J is too far from unitary
cudaError_t launch_lowdin_j(Dims* dims, const ProbPtr* ptrs, int batch, int l, int cond, cudaStream_t st);
cudaError_t launch_oz_range(int stage, const Dims* dims, const ProbPtr* ptrs, int batch, const Caps& cap,
                            const OzScratch& sc, int chunk, int cond, int* err, cudaStream_t st);

// Cholesky QR (two passes) of B^H for well-conditioned instances, Householder
// for the others (cholqr.cu); writes dims[p].qflag.  oz: the products on the
// tensor cores (raising *err on a pipeline stall), or null for double-float
// GEMMs.  phases: with the column phases of the Householder QR (with oz only).
cudaError_t run_cholqr_bh(Dims* dims, const ProbPtr* ptrs, int batch, const Caps& cap, cudaStream_t st,
                          const OzScratch* oz, int* err, bool phases);
cudaError_t cholqr_prepare();
cudaError_t launch_oz_digits_theta(const Dims* dims, const ProbPtr* ptrs, uint16_t* Bd, int* Bs, int m, int n,
                                   int batch, cudaStream_t st);
// (Q_f's digits in Ad / As from launch_oz_digits_qf)
cudaError_t launch_proj_oz(const Dims* dims, const ProbPtr* ptrs, const uint16_t* Ad, const int* As,
                           const uint16_t* Bd, const int* Bs, int m, int n, int l, int batch, int* err,
                           cudaStream_t st);
// Digits of Q_f (the projection's left operand, conjugated by the MMAs; Q_f's
// entries are rounded to what its four digits hold, or where theta's rows are
// graded take seven as they are) into Ad (room for seven) / As, and the
// Gram matrix E = Q_f^H Q_f - I of the re-orthonormalisation from them into
// ptrs[z].R (l x l column-major), FP64-accurate, on the tensor cores.
cudaError_t launch_oz_digits_qf(const Dims* dims, const ProbPtr* ptrs, float2* Qf, uint16_t* Ad, int* As, int m, int l, int batch,
                                cudaStream_t st);
cudaError_t launch_oz_gram(const Dims* dims, const ProbPtr* ptrs, const uint16_t* Ad, const int* As, int m, int l,
                           int batch, int* err, cudaStream_t st);

// Launch choices of the mixed form that the autotuner may override (0 keeps
// each size rule): tc_half = 1 splits the tensor-core products' columns over
// two CTAs; qr_threads sets the CTA size of the blocked FP32 Householder QRs
// (128, 256, 512) and takes them in place of the Cholesky QR; qrbh forces the
// QR of B^H (1 one-CTA Householder, 2 many-CTA Householder, 3 Cholesky QR with
// Householder for ill-conditioned instances, mixed_qrbh's rule); jac the
// Jacobi SVD (1 the one-CTA FP64 kernel, 2 the cluster form, 3 the one-CTA
// double-float one); dfg the products after the projection: on the tensor
// cores from digit splits (0 by size, 1) or as double-float CUDA-core GEMMs (2).
struct MixedKnobs {
  int tc_half, qr_threads, qrbh, jac, dfg;
};

// The choices a launch on `batch` problems of capacities cap makes (a set knob,
// or the size rule): the QR of B^H (1, 2 or 3; 4 is 3 with Householder's column
// phases) and the Jacobi SVD.
int mixed_qrbh(const MixedKnobs& kn, const Caps& cap, int batch);
int mixed_jac(const MixedKnobs& kn, const Caps& cap, int batch);

// Everything that must happen outside a stream capture before
// run_rrsvd_mixed runs on capacities `cap` (shared-memory limits, the
// tensor-map encoder entry point).
cudaError_t mixed_prepare(const Caps& cap);
cudaError_t qr_blocked_prepare(int M, int N, int L);

// Alg. 1 with tensor-core products and the FP64-accurate projection / FP64
// small SVD.  The FP32 arrays are laid out at the capacities `cap` (the
// maxima over the batch, which size mixed_sizes/mixed_carve); each instance
// uses its own (m, n, k, l) from dims, zero-padded up to them.  Instance z
// draws Omega from chain chain0 + z chain_stride at `sweep`, or, with
// chain_stride < 0, from its own chain index at *sweep_dev.
cudaError_t run_rrsvd_mixed(const Dims* dims, const ProbPtr* ptrs, int batch, const Caps& cap, const MixedPtrs& mp,
                            int q, uint64_t seed, uint64_t sweep, int64_t chain0, int chain_stride, int* status,
                            int* err, cudaStream_t st, const uint64_t* sweep_dev = nullptr,
                            const MixedKnobs* knobs = nullptr, int bf16 = 0);

}  // namespace tg
