// TEBD two-site update kernels, plain FP64 (sm_103a): theta contraction with
// the gate fused in its epilogue, the per-sweep size plan, the Vidal-form
// rebuild after truncation, and one-site expectation values.
#include <cuda_runtime.h>
#include <math.h>

#include "internal.cuh"
#include "once.cuh"
#include "profiler.cuh"
#include "stages.cuh"

namespace tg {

// ---------------------------------------------------------------------------
// Sizes of every bond of a wave from the current bond dimensions:
//   m = d_b chi_{b-1}, n = d_{b+1} chi_{b+1}, k = min(cap_b, m, n),
//   l = min(k + p, m, n)   (sketch width; exact when it reaches min(m, n)).
// Bonds of one parity share no site, so their updates are independent.
// ---------------------------------------------------------------------------
__global__ void k_plan(const ProbPtr* __restrict__ ptrs, Dims* dims, int batch, int p, int digits) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= batch) return;
  dims[t] = plan_dev(ptrs[t], p, digits);
}

cudaError_t launch_plan(const ProbPtr* ptrs, Dims* dims, int batch, int p, cudaStream_t st, int digits) {
  ProfScope ps("k_plan", st);
  k_plan<<<(batch + 127) / 128, 128, 0, st>>>(ptrs, dims, batch, p, digits);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// theta~ of each bond (Eq. deftheta then Eq. defupdatetheta):
//   C[(i',a),(j',c)] = sum_g (lam_l[a] Gl[i'][a][g] lam_m[g]) (Gr[j'][g][c] lam_r[c])
//   theta~[i*cl + a][j*cr + c] = sum_{i'j'} G[(i dr + j), (i' dr + j')] C[(i',a),(j',c)]
// A CTA owns an (alpha, beta) block with every i, j (the gate mixes only the
// physical indices), so the gate is applied from shared memory right after
// the contraction.  Tile: dl*TA <= 32 rows (TA >= 1), dr*TB <= 32 columns.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_theta(const Dims* __restrict__ dims, const ProbPtr* __restrict__ ptrs,
                                               int identity_gate, int skip_pre, int skip_dig) {
  extern __shared__ cplx th_sm[];
  const int p = blockIdx.z;
  const Dims D = dims[p];
  if (!D.active) return;
  const ProbPtr P = ptrs[p];
  if (skip_pre && !identity_gate && P.Cpre) return;  // contracted by launch_theta_df
  if (skip_dig && !P.Cpre && (D.dig || skip_dig == 2) && theta_digits_rule(D.m, D.n, D.cm)) return;  // k_gate_small's
  theta_tile_dev(D, P, blockIdx.y, blockIdx.x, identity_gate, th_sm);
}

// theta <- gate applied to the contraction in theta, in place, for the bonds
// k_theta leaves to the digit-split contraction: a thread takes the d_l d_r
// entries (i, j) of one (alpha, beta), which no other thread touches, through
// shared memory.  Bound by the FP64
// pipe, (d_l d_r)^2 complex multiply-adds per (alpha, beta): 12 chains' bonds
// of chi up to 128, contraction and gate: 8.3 ms on the FP64 pipe alone, 2.1 ms
// with this and the digits (0.6 the contraction, 1.1 both kernels' rest).
enum { GS_T = 128 };

__global__ void __launch_bounds__(GS_T) k_gate_small(const Dims* __restrict__ dims,
                                                     const ProbPtr* __restrict__ ptrs, int need_dig) {
  extern __shared__ cplx gs_sm[];  // [dd][GS_T], then the gate
  const int p = blockIdx.y;
  const Dims D = dims[p];
  if (!D.active || (need_dig && !D.dig) || !theta_digits_rule(D.m, D.n, D.cm)) return;
  const ProbPtr P = ptrs[p];
  if (P.Cpre) return;
  const int dl = D.dl, dr = D.dr, cl = D.cl, cr = D.cr, dd = dl * dr, tid = threadIdx.x;
  cplx* g = gs_sm + (size_t)dd * GS_T;
  for (int e = tid; e < dd * dd; e += GS_T) g[e] = P.gate[e];
  __syncthreads();
  const int64_t n = (int64_t)cl * cr;
  cplx* th = const_cast<cplx*>(P.theta);
  for (int64_t e = (int64_t)blockIdx.x * GS_T + tid; e < n; e += (int64_t)gridDim.x * GS_T) {
    const int al = (int)(e / cr), be = (int)(e % cr);
    cplx* t0 = th + (int64_t)al * D.n + be;
    for (int k = 0; k < dd; ++k) gs_sm[k * GS_T + tid] = t0[(int64_t)(k / dr) * cl * D.n + (k % dr) * cr];
    for (int r = 0; r < dd; ++r) {
      cplx v = cmk(0.0, 0.0);
      for (int k = 0; k < dd; ++k) cfma(v, g[r * dd + k], gs_sm[k * GS_T + tid]);
      t0[(int64_t)(r / dr) * cl * D.n + (r % dr) * cr] = v;
    }
  }
}

static size_t gs_smem(int dd) { return sizeof(cplx) * ((size_t)dd * GS_T + (size_t)dd * dd); }

static const size_t TH_SMEM = sizeof(cplx) * (2 * TH_TK * TH_MAXR + TH_MAXR * TH_MAXR);

cudaError_t theta_prepare() {
  static DeviceOnce once;
  return once([] {
    const cudaError_t e = cudaFuncSetAttribute(k_gate_small, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                               (int)gs_smem(GATE_GEMM_MIN - 1));
    return e != cudaSuccess ? e
                            : cudaFuncSetAttribute(k_theta, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TH_SMEM);
  });
}

cudaError_t launch_gate_small(const Dims* dims, const ProbPtr* ptrs, int batch, const Caps& cap, int need_dig,
                              cudaStream_t st) {
  // (cap.dl cap.dr may come from different bonds; those of GATE_GEMM_MIN and more have their own path)
  const int dd = cap.dl * cap.dr < GATE_GEMM_MIN ? cap.dl * cap.dr : GATE_GEMM_MIN - 1;
  const cudaError_t e = theta_prepare();
  if (e != cudaSuccess) return e;
  ProfScope ps("k_theta", st);
  size_t gx = ((size_t)cap.cl * cap.cr + GS_T - 1) / GS_T;
  const size_t most = (8 * 152 * 8 + batch - 1) / batch;
  gx = gx > most ? most : gx;
  k_gate_small<<<dim3((unsigned)gx, batch), GS_T, gs_smem(dd), st>>>(dims, ptrs, need_dig);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Gate as a GEMM (Eq. defupdatetheta for large local dimensions):
//   theta~[(i cl + a), (j cr + c)] = sum_{i'j'} G[(i dr + j), (i' dr + j')] C[(i' cl + a), (j' cr + c)],
// rows (i, j) of G times the (d_l d_r) x (cl cr) matrix whose column (a, c)
// gathers C over the physical indices.  32 x 32 output tiles (rows (i, j),
// columns (a, c) with c fastest), 2 x 2 outputs per thread, K = d_l d_r in
// slices of 16, FP64 (the layout of k_zgemm).
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_gate_gemm(const Dims* __restrict__ dims, const ProbPtr* __restrict__ ptrs) {
  constexpr int T = 32, TK = 16;
  __shared__ cplx As[TK][T + 1];  // G[row][k]
  __shared__ cplx Bs[TK][T + 1];  // C-gather[k][col]
  const int p = blockIdx.z;
  const Dims D = dims[p];
  if (!D.active) return;
  const ProbPtr P = ptrs[p];
  if (!P.Cpre) return;
  const int dl = D.dl, dr = D.dr, cl = D.cl, cr = D.cr;
  const int M = dl * dr, N = cl * cr, K = M;
  const int tm = blockIdx.y * T, tn = blockIdx.x * T;
  if (tm >= M || tn >= N) return;
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  const int n_ = D.n;
  cplx acc[2][2];
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 2; ++j) acc[i][j] = cmk(0.0, 0.0);
  for (int k0 = 0; k0 < K; k0 += TK) {
    for (int e = tid; e < T * TK; e += 256) {  // G tile: consecutive threads along k (contiguous)
      const int kk = e % TK, r = e / TK;
      const int gr = tm + r, gk = k0 + kk;
      As[kk][r] = (gr < M && gk < K) ? P.gate[(int64_t)gr * K + gk] : cmk(0.0, 0.0);
    }
    for (int e = tid; e < T * TK; e += 256) {  // C tile: consecutive threads along (a, c), c fastest
      const int c = e % T, kk = e / T;
      const int gn = tn + c, gk = k0 + kk;
      cplx v = cmk(0.0, 0.0);
      if (gn < N && gk < K) {
        const int ip = gk / dr, jp = gk % dr, a = gn / cr, cc = gn % cr;
        v = P.Cpre[(int64_t)(ip * cl + a) * n_ + jp * cr + cc];
      }
      Bs[kk][c] = v;
    }
    __syncthreads();
#pragma unroll 4
    for (int kk = 0; kk < TK; ++kk) {
      const cplx a0 = As[kk][ty], a1 = As[kk][ty + 16];
      const cplx b0 = Bs[kk][tx], b1 = Bs[kk][tx + 16];
      cfma(acc[0][0], a0, b0);
      cfma(acc[0][1], a0, b1);
      cfma(acc[1][0], a1, b0);
      cfma(acc[1][1], a1, b1);
    }
    __syncthreads();
  }
  cplx* th = const_cast<cplx*>(P.theta);
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const int r = tm + ty + 16 * i, c = tn + tx + 16 * j;
      if (r < M && c < N) {
        const int ii = r / dr, jj = r % dr, a = c / cr, cc = c % cr;
        th[(int64_t)(ii * cl + a) * n_ + jj * cr + cc] = acc[i][j];
      }
    }
}

cudaError_t launch_gate_gemm(const Dims* dims, const ProbPtr* ptrs, int batch, const Caps& cap, cudaStream_t st) {
  const int M = cap.dl * cap.dr, N = cap.cl * cap.cr;
  if (M < GATE_GEMM_MIN) return cudaSuccess;  // no bond of this wave takes the GEMM path
  ProfScope ps("k_gate_gemm", st);
  dim3 grid((N + 31) / 32, (M + 31) / 32, batch);
  k_gate_gemm<<<grid, 256, 0, st>>>(dims, ptrs);
  return cudaGetLastError();
}

cudaError_t launch_theta(const Dims* dims, const ProbPtr* ptrs, int batch, const Caps& cap, cudaStream_t st,
                         int identity_gate, int skip_pre, int skip_dig) {
  const int TA = (cap.dl >= 32) ? 1 : 32 / cap.dl;
  const int TB = (cap.dr >= 32) ? 1 : 32 / cap.dr;
  dim3 grid((cap.cr + TB - 1) / TB, (cap.cl + TA - 1) / TA, batch);
  const cudaError_t e = theta_prepare();
  if (e != cudaSuccess) return e;
  ProfScope ps("k_theta", st);
  k_theta<<<grid, 256, TH_SMEM, st>>>(dims, ptrs, identity_gate, skip_pre, skip_dig);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Rebuild after truncation (Eq. defdiscweigt and the Vidal extraction):
//   chi' = #{i < k : s_i > cutoff s_1}, lambda'[b] = s / ||s_kept||,
//   w = 1 - sum_kept s^2 / ||theta~||_F^2,
//   Gamma'[b]^i[a][g]   = U[(i*cl + a)][g] / lam_l[a],
//   Gamma'[b+1]^j[g][c] = Vh[g][(j*cr + c)] / lam_r[c]   (divide only if lam > 0).
// A zero or non-finite theta~ leaves the bond unchanged and raises status bit
// 1.  Memory-bound on many CTAs per bond (one per RB_ELEMS elements of the
// larger Gamma, four waves of CTAs at most); on one CTA per bond the 15 bonds
// of a spin-boson wave of local dimension 32 and chi 256 took 7 ms.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_rebuild(const Dims* __restrict__ dims, const ProbPtr* __restrict__ ptrs,
                                                 double cutoff, double* wout, int* status) {
  __shared__ int s_rank;
  __shared__ double s_inv;
  const int p = blockIdx.x;
  const Dims D = dims[p];
  if (!D.active) return;
  rebuild_dev(D, ptrs[p], cutoff, wout + p, status, &s_rank, &s_inv, blockIdx.y, gridDim.y);
}

enum { RB_ELEMS = 4096 };

cudaError_t launch_rebuild(const Dims* dims, const ProbPtr* ptrs, int batch, const Caps& cap, double cutoff,
                           double* wout, int* status, cudaStream_t st) {
  ProfScope ps("k_rebuild", st);
  const size_t elems = (size_t)(cap.m > cap.n ? cap.m : cap.n) * cap.k;
  size_t parts = (elems + RB_ELEMS - 1) / RB_ELEMS;
  const size_t most = (4 * 152 * 8 + batch - 1) / batch;
  parts = parts > most ? most : parts;
  k_rebuild<<<dim3(batch, (unsigned)parts), 256, 0, st>>>(dims, ptrs, cutoff, wout, status);
  return cudaGetLastError();
}

// Adds the discarded weights of a wave, in problem order, into the per-chain
// accumulators wacc[2 slot] (sum of w) and wacc[2 slot + 1] (product of 1 - w).
__global__ void k_wacc(const Dims* dims, const ProbPtr* ptrs, const double* wout, int batch, double* wacc) {
  for (int p = 0; p < batch; ++p) {
    if (!dims[p].active) continue;
    const int s = ptrs[p].slot;
    wacc[2 * s] += wout[p];
    wacc[2 * s + 1] *= (1.0 - wout[p]);
    if (ptrs[p].wbond) *ptrs[p].wbond = wout[p];
  }
}

cudaError_t launch_wacc(const Dims* dims, const ProbPtr* ptrs, const double* wout, int batch, double* wacc,
                        cudaStream_t st) {
  k_wacc<<<1, 1, 0, st>>>(dims, ptrs, wout, batch, wacc);
  return cudaGetLastError();
}

// The sweep counter of the Philox sketch lives on the device so that a
// captured sweep can be replayed.
__global__ void k_sweep_tick(uint64_t* sweep_dev) { *sweep_dev += 1; }

cudaError_t launch_sweep_tick(uint64_t* sweep_dev, cudaStream_t st) {
  k_sweep_tick<<<1, 1, 0, st>>>(sweep_dev);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// <O_site> = sum_{a,c} lam_l[a]^2 lam_r[c]^2 sum_{i,i'} conj(G^i[a][c]) O[i][i'] G^{i'}[a][c]
// FP64-pipe bound (4 d^2 multiply-adds per element of the bond pair): the
// elements are cut into EX_PARTS fixed chunks (partial sums the same whatever
// the grid), a CTA takes the chunks p = blockIdx, blockIdx + gridDim, ..., and
// the last kernel adds the partials in order.  Spread over the chip, a site
// with d = 32 and bonds of 256 takes ~0.6 ms instead of 70 ms on one SM, one
// with d = 3 and bonds of 128 ~12 us instead of 130 us; a small site (under
// EX_SMALL elements x d^2) stays one launch of one CTA.
// ---------------------------------------------------------------------------
enum { EX_SMALL = 16384 };

__global__ void __launch_bounds__(256) k_expect(ChainDev ch, int site, const cplx* __restrict__ op, int d,
                                                cplx* part, cplx* out) {
  __shared__ double red[32];
  const int cl = ch.chi_ext[site], cr = ch.chi_ext[site + 1];
  const int capl = ch.cap_ext[site], capr = ch.cap_ext[site + 1];
  const double* ll = ch.lam_ext[site];
  const double* lr = ch.lam_ext[site + 1];
  const cplx* G = ch.gamma[site];
  const int64_t total = (int64_t)cl * cr;
  const int nchunk = out ? 1 : EX_PARTS;
  const int64_t len = (total + nchunk - 1) / nchunk;
  for (int p = blockIdx.x; p < nchunk; p += gridDim.x) {
    double sr = 0.0, si = 0.0;
    const int64_t e1 = min(total, len * (p + 1));
    for (int64_t e = len * p + threadIdx.x; e < e1; e += blockDim.x) {
      const int a = (int)(e / cr), c = (int)(e % cr);
      const double wgt = ll[a] * ll[a] * lr[c] * lr[c];
      for (int i = 0; i < d; ++i) {
        const cplx gi = G[((int64_t)i * capl + a) * capr + c];
        cplx og = cmk(0.0, 0.0);
        for (int ip = 0; ip < d; ++ip) cfma(og, op[i * d + ip], G[((int64_t)ip * capl + a) * capr + c]);
        cplx t = cmk(0.0, 0.0);
        cfma_conj(t, gi, og);
        sr += wgt * t.x;
        si += wgt * t.y;
      }
    }
    sr = block_sum(sr, red);
    si = block_sum(si, red);
    if (threadIdx.x == 0) *(out ? out : part + p) = cmk(sr, si);
  }
}

__global__ void k_expect_sum(const cplx* __restrict__ part, cplx* out) {
  const int lane = threadIdx.x;
  cplx s = cmk(0.0, 0.0);
  for (int p = lane; p < EX_PARTS; p += 32) s = cadd(s, part[p]);
  s = warp_sum(s);
  if (lane == 0) *out = s;
}

// The handle's flags, and n doubles of src (with chi: an int too), into pinned
// host memory: a query reads its answer after one launch and one wait.  (Each
// copy to pageable memory is a wait of its own: an expectation value took 40
// us with them, 15 with this; the two kernels themselves take 20 of a large
// site's.)
__global__ void k_report(const int* __restrict__ status, const int* __restrict__ tcerr, const double* __restrict__ src,
                         int n, const int* __restrict__ chi, int* head, double* out) {
  for (int i = threadIdx.x; i < n; i += blockDim.x) out[i] = src[i];
  if (threadIdx.x == 0) {
    head[0] = *status;
    head[1] = tcerr ? *tcerr : 0;
    head[2] = chi ? *chi : 0;
  }
}

cudaError_t launch_report(const int* status, const int* tcerr, const double* src, int n, const int* chi, int* head,
                          double* out, cudaStream_t st) {
  k_report<<<1, n > 32 ? 128 : 32, 0, st>>>(status, tcerr, src, n, chi, head, out);
  return cudaGetLastError();
}

cudaError_t launch_expect(const ChainDev& ch, int site, int64_t elems, const cplx* op, int d, cplx* part, cplx* out,
                          cudaStream_t st) {
  ProfScope ps("k_expect", st);
  if (elems * d * d <= EX_SMALL) {
    k_expect<<<1, 256, 0, st>>>(ch, site, op, d, part, out);
  } else {
    k_expect<<<EX_PARTS, 256, 0, st>>>(ch, site, op, d, part, nullptr);
    k_expect_sum<<<1, 32, 0, st>>>(part, out);
  }
  return cudaGetLastError();
}

}  // namespace tg
