// Q = Y J of the FP32 Cholesky QR (sm_103a): Y (M x l complex FP32 per
// instance) times the upper triangular J = S R^-1, FP32 throughout.
//
// A CTA takes 64 rows and goes through the columns 64 at a time from the right
// to the left, so that src and dst may be the same array: column tile t needs
// the columns up to its own end, and those right of it are done.  256 threads,
// 4 x 4 complex results each, 16 deep per shared-memory tile, the next tile in
// registers meanwhile: 64 multiply-adds for four 16-byte shared loads, bound
// by the FP32 pipe.  152 x 2000 x 120: 0.37 ms at the pipe's rate, against
// 1.5 ms for the same product from 28 digit pairs (whose MMAs are as many for
// four digits, and whose results are scaled in FP64).
#include <cuda_runtime.h>

#include "internal.cuh"
#include "mixed.cuh"
#include "profiler.cuh"

namespace tg {

enum { TR_B = 64, TR_K = 16 };

__global__ void __launch_bounds__(256) k_trmm_f32(const float2* src, float2* dst, const Dims* __restrict__ dims,
                                                  const ProbPtr* __restrict__ ptrs, int Mc, int Lc, int use_n,
                                                  int pass) {
  __shared__ __align__(16) float2 sa[TR_K][TR_B], sb[TR_K][TR_B + 2];
  const int z = blockIdx.y;
  const Dims D = dims[z];
  if (!D.active || D.cf || D.cq < pass) return;
  const int M = use_n ? D.n : D.m, L = D.l, r0 = blockIdx.x * TR_B;
  const float2* X = src + (size_t)z * Mc * Lc;
  float2* Q = dst + (size_t)z * Mc * Lc;
  const float2* J = reinterpret_cast<const float2*>(ptrs[z].J);  // column-major L x L
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  for (int c0 = (L - 1) / TR_B * TR_B; c0 >= 0; c0 -= TR_B) {
    float2 acc[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) acc[i][j] = make_float2(0.f, 0.f);
    const int kend = min(L, c0 + TR_B);
    float2 ra[4], rb[4];
    auto fetch = [&](int k0) {
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int r = r0 + (tid & 63), k = k0 + (tid >> 6) + 4 * i;
        ra[i] = (r < M && k < kend) ? X[(size_t)k * Mc + r] : make_float2(0.f, 0.f);
        const int c = c0 + ty + 16 * i, kb = k0 + tx;
        rb[i] = (c < L && kb <= c) ? J[(size_t)c * L + kb] : make_float2(0.f, 0.f);
      }
    };
    fetch(0);
    for (int k0 = 0; k0 < kend; k0 += TR_K) {
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        sa[(tid >> 6) + 4 * i][tid & 63] = ra[i];
        sb[tx][ty + 16 * i] = rb[i];
      }
      __syncthreads();
      if (k0 + TR_K < kend) fetch(k0 + TR_K);
#pragma unroll
      for (int k = 0; k < TR_K; ++k) {
        float2 u[4], v[4];  // rows 2 tx, 2 tx + 1 (+ 32), columns 2 ty, 2 ty + 1 (+ 32)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const float4 p = *reinterpret_cast<const float4*>(&sa[k][2 * tx + 32 * h]);
          u[2 * h] = make_float2(p.x, p.y);
          u[2 * h + 1] = make_float2(p.z, p.w);
          const float4 q = *reinterpret_cast<const float4*>(&sb[k][2 * ty + 32 * h]);
          v[2 * h] = make_float2(q.x, q.y);
          v[2 * h + 1] = make_float2(q.z, q.w);
        }
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            acc[i][j].x = fmaf(u[i].x, v[j].x, fmaf(-u[i].y, v[j].y, acc[i][j].x));
            acc[i][j].y = fmaf(u[i].x, v[j].y, fmaf(u[i].y, v[j].x, acc[i][j].y));
          }
      }
      __syncthreads();
    }
    // rows past the instance's own become zero, as in the array read
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int c = c0 + 2 * ty + (j & 1) + 32 * (j >> 1);
      if (c >= L) continue;
#pragma unroll
      for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          const int r = r0 + 2 * tx + 32 * h + i;
          if (r < Mc) Q[(size_t)c * Mc + r] = r < M ? acc[2 * h + i][j] : make_float2(0.f, 0.f);
        }
    }
    // (the barrier after the last k tile: every thread has read its columns)
  }
}

cudaError_t launch_trmm_f32(const float2* src, float2* dst, const Dims* dims, const ProbPtr* ptrs, int Mc, int Lc,
                            int use_n, int pass, int batch, cudaStream_t st) {
  ProfScope ps("k_trmm_f32", st);
  k_trmm_f32<<<dim3((Mc + TR_B - 1) / TR_B, batch), 256, 0, st>>>(src, dst, dims, ptrs, Mc, Lc, use_n, pass);
  return cudaGetLastError();
}

}  // namespace tg
