// Householder QR with explicit Q of small FP64 matrices (sm_103a), one
// thread-block cluster per matrix, the matrix in shared memory.
//
// The arithmetic is qr_dev's (stages.cuh), bit for bit, whatever the cluster
// size.  Every CTA of the cluster holds the whole M x L array and forms every
// reflector itself (warp 0: H_j applied to column j + 1, then its reflector):
// the chain then has no exchange in it.  The columns right of j + 1 are dealt
// out round robin; the owner of column j + 2 applies H_j to it first and
// stores it into every CTA's array through distributed shared memory, while
// the chain still works on column j + 1; one cluster barrier per column.  Q's
// columns need all reflectors and nothing else, one warp each.
//
// What bounds it: the chain, about 50 FP64 instructions of 64 clocks for
// 64 rows; without a cluster (no idle SMs) the FP64 pipe.  Cluster size: as
// many SMs as the batch leaves idle, up to eight.  Measured, QR and Q: 10 x
// 64 x 42 583 us on one CTA of 1024 threads each with the matrix in global
// memory, 146 us here; 256 x 64 x 42 1.49 ms against 0.68 (FP64 pipe 85% busy);
// one 96 x 18 212 us against 97.
#include <cooperative_groups.h>
#include <cuda_runtime.h>
#include <math.h>

#include "internal.cuh"
#include "once.cuh"
#include "profiler.cuh"
#include "stages.cuh"

namespace cg = cooperative_groups;

namespace tg {

enum { QS_MAXCL = 8, QS_MAXL = 160, QS_THREADS = 512, QS_CL_THREADS = 128 };
static const size_t QS_SMEM = 200 * 1024;

template <int QS>
__global__ void __launch_bounds__(QS_THREADS) k_qr_small(const Dims* __restrict__ dims,
                                                         const ProbPtr* __restrict__ ptrs, int which) {
  extern __shared__ __align__(16) unsigned char qs_raw[];
  __shared__ double tau[QS_MAXL];
  __shared__ cplx alph[QS_MAXL];
  cg::cluster_group cluster = cg::this_cluster();
  const int CL = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
  const int p = blockIdx.x / CL;
  const Dims D = dims[p];
  if (!D.active || !qr_takes(D, which)) return;  // uniform over the cluster
  const ProbPtr& P = ptrs[p];
  const int M = (QS == QR_Y) ? D.m : D.n, L = D.l;
  const cplx* A = (QS == QR_Y) ? P.Y : P.Yt;
  cplx* Qo = (QS == QR_Y) ? P.Q : P.Qt;
  cplx* V = reinterpret_cast<cplx*>(qs_raw);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = blockDim.x >> 5;
  const int gl = lane & (QR_G - 1), half = lane / QR_G;
  const unsigned gmask = ((1u << QR_G) - 1u) << (lane & ~(QR_G - 1));
  const int slot = qr_slot(warp);
  for (int e = tid; e < M * L; e += blockDim.x) V[e] = A[e];
  __syncthreads();
  if (warp == 0) qr_reflect<QS == QR_BH>(V, 0, qr_norm2(V, 0, M, lane), lane, tau, alph);
  if (CL > 1) cluster.sync();  // every CTA runs, with the whole array, before any column is sent
  else __syncthreads();
  for (int j = 0; j + 1 < L; ++j) {
    const double t = tau[j];
    const cplx* v = V + j * M;
    if (warp == 0) {
      qr_next<QS == QR_BH>(v, V + (j + 1) * M, j, M, t, lane, tau + j + 1, alph + j + 1);
    } else {
      // the own columns from j + 2 on, c = rank mod CL
      const int c0 = j + 2 + (rank - (j + 2) % CL + CL) % CL;
      if (t != 0.0)
        for (int c = c0 + (2 * slot + half) * CL; c < L; c += 2 * (nw - 1) * CL)
          qr_apply(v, V + c * M, j, M, t, gl, gmask);
      if (CL > 1 && slot == 0 && c0 == j + 2 && c0 < L) {  // done by this warp: the next step's chain needs it
        __syncwarp();
        const cplx* a = V + c0 * M;
        for (int o = 1; o < CL; ++o) {
          cplx* d = cluster.map_shared_rank(V, (rank + o) % CL) + c0 * M;
          for (int r = lane; r < M; r += 32) d[r] = a[r];
        }
      }
    }
    if (CL > 1) cluster.sync();
    else __syncthreads();
  }
  if (QS == QR_BH) {  // X = Rb^H (see qr_dev); every CTA holds all of Rb
    for (int e = rank * blockDim.x + tid; e < L * L; e += CL * blockDim.x) {
      const int c = e / L, r = e % L;
      cplx x = cmk(0.0, 0.0);
      if (c < r) x = cconj(V[r * M + c]);
      else if (c == r) x = cconj(alph[c]);
      P.R[e] = x;
    }
  }
  for (int i = warp * CL + rank; i < L; i += nw * CL) {
    const int c = L - 1 - i;
    qr_qcol(V, tau, Qo + (int64_t)c * M, c, M, lane);
  }
}

bool qr_small_fits(int stage, const Caps& cap) {
  const size_t M = (stage == QR_Y) ? cap.m : cap.n;
  return cap.l <= QS_MAXL && M * (size_t)cap.l * sizeof(cplx) <= QS_SMEM;
}

template <int QS>
static cudaError_t qs_attr() {
  return cudaFuncSetAttribute(k_qr_small<QS>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)QS_SMEM);
}

cudaError_t qr_small_prepare() {
  static DeviceOnce once;
  return once([] {
    for (cudaError_t e : {qs_attr<QR_Y>(), qs_attr<QR_YT>(), qs_attr<QR_BH>()})
      if (e != cudaSuccess) return e;
    return cudaSuccess;
  });
}

cudaError_t launch_qr_small(int stage, const Dims* dims, const ProbPtr* ptrs, int batch, const Caps& cap,
                            cudaStream_t st, int which) {
  cudaError_t e = qr_small_prepare();
  if (e != cudaSuccess) return e;
  const int M = (stage == QR_Y) ? cap.m : cap.n;
  int cl = 1;
  while (cl < QS_MAXCL && batch * cl * 2 <= 152 && cl * 4 <= cap.l) cl *= 2;
  const int nt = cl > 2 || cap.l < 16 ? QS_CL_THREADS : QS_THREADS;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(batch * cl);
  cfg.blockDim = dim3(nt);
  cfg.dynamicSmemBytes = sizeof(cplx) * (size_t)M * cap.l;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = cl;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  switch (stage) {
    case QR_Y: return cudaLaunchKernelEx(&cfg, k_qr_small<QR_Y>, dims, ptrs, which);
    case QR_YT: return cudaLaunchKernelEx(&cfg, k_qr_small<QR_YT>, dims, ptrs, which);
    case QR_BH: return cudaLaunchKernelEx(&cfg, k_qr_small<QR_BH>, dims, ptrs, which);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace tg
