// Inverses of the unit-lower diagonal blocks L_JJ (complex FP32), built once per factorization so
// that the solve applies every diagonal block as one product (y_J = L_JJ^{-1} r_J) instead of a
// sequential chain over its tiles.  With the tile inverses Linv_tt of the factorization:
//   Inv(t', t') = Linv_t't',   Inv(t, t') = -Linv_tt * sum_{s=t'}^{t-1} L(t, s) Inv(s, t')   (t > t').
// One thread block per (block J, tile column t') forms Inv(t, t') for t = t'+1, ..., nt-1 in order
// (each needs the ones above it in the same column).  Tiles are b x b, row-major, b in {64, 128}.
// Every tile is also stored transposed, InvT(t', t) = Inv(t, t')^T (t >= t', diagonal included),
// so that the backward solve streams contiguous row strips as well.
// The columns of an inverse are independent, so a thread block takes one 64-column strip of a tile column (half
// the chain for one block, twice the blocks, two of them on an SM).  Products: shared-memory staged FP32 SIMT GEMM,
// each of the 256 threads owning (b / 16) x 4 entries, the columns 16 apart (conflict-free), the next 16 of K
// in flight in registers.  Bound by FP32 FMAs (a product of 128-tiles is 4.2e6 complex ones, 32 us of an SM); 112
// blocks of 512: 1.00 -> 0.58 ms (0.38 at the FMA rate) against whole tile columns of 8 x 8 entries a thread.
#include <cuda_runtime.h>

#include "device.cuh"
#include "kernels.h"

namespace d3m {

namespace {

constexpr int IT = 256;   // threads
constexpr int KC = 16;    // k-chunk of the staged products
constexpr int CW = 64;    // columns of a strip
constexpr int LDC = CW + 1;

// acc += A * Y for a b x b tile A in global memory (row-major) and b rows of CW columns Y: in global memory (leading
// dimension B; GLOBAL) or in shared memory (LDC)
template <int B, bool GLOBAL>
__device__ __forceinline__ void gemm_strip(const float2* __restrict__ A, const float2* Y, float2* sA, float2* sB,
                                           float2 (&acc)[B / 16][4]) {
  constexpr int TM = B / 16, LDA = B + 2, NA = B * KC / IT, NB = KC * CW / IT;
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  float2 ra[NA], rb[NB];
  auto fetch = [&](int k0) {
#pragma unroll
    for (int i = 0; i < NA; ++i) ra[i] = A[(int64_t)((tid >> 4) + i * (IT / KC)) * B + k0 + (tid & 15)];
    if constexpr (GLOBAL) {
#pragma unroll
      for (int i = 0; i < NB; ++i) rb[i] = Y[(int64_t)(k0 + (tid >> 6) + i * (IT / CW)) * B + (tid & 63)];
    }
  };
  fetch(0);
#pragma unroll 1
  for (int k0 = 0; k0 < B; k0 += KC) {
    __syncthreads();                                   // the previous chunk is consumed
#pragma unroll
    for (int i = 0; i < NA; ++i) sA[(tid & 15) * LDA + (tid >> 4) + i * (IT / KC)] = ra[i];   // transposed: (k, row)
    if constexpr (GLOBAL) {
#pragma unroll
      for (int i = 0; i < NB; ++i) sB[((tid >> 6) + i * (IT / CW)) * CW + (tid & 63)] = rb[i];
    }
    __syncthreads();
    if (k0 + KC < B) fetch(k0 + KC);
#pragma unroll 2
    for (int kk = 0; kk < KC; ++kk) {
      float2 a[TM], bb[4];
#pragma unroll
      for (int i = 0; i < TM; i += 2) {
        const float4 v = *reinterpret_cast<const float4*>(sA + kk * LDA + ty * TM + i);
        a[i] = make_float2(v.x, v.y);
        a[i + 1] = make_float2(v.z, v.w);
      }
#pragma unroll
      for (int j = 0; j < 4; ++j) bb[j] = GLOBAL ? sB[kk * CW + tx + 16 * j] : Y[(k0 + kk) * LDC + tx + 16 * j];
#pragma unroll
      for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = cfma(a[i], bb[j], acc[i][j]);
    }
  }
}

template <int B>
__global__ void __launch_bounds__(IT, 2) inv_build_kernel(const int2* __restrict__ work, const int32_t* __restrict__ tstart,
                                                          const int64_t* __restrict__ tcolptr,
                                                          const int64_t* __restrict__ inv_off,
                                                          const int64_t* __restrict__ invT_off,
                                                          const float2* __restrict__ L, const float2* __restrict__ Linv,
                                                          float2* Inv, float2* __restrict__ InvT) {
  constexpr int TM = B / 16, LDA = B + 2;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float2* sA = reinterpret_cast<float2*>(smem_raw);   // [KC][LDA]
  float2* sB = sA + KC * LDA;                          // [KC][CW]
  float2* sC = sB + KC * CW;                           // [B][LDC]
  constexpr int NS = B / CW;                           // strips of a tile column
  const int2 wk = work[blockIdx.x / NS];
  const int k = wk.x, tq = wk.y, cs = (int)(blockIdx.x % NS) * CW;
  const int t0 = tstart[k], nt = tstart[k + 1] - t0;
  const int64_t ib = inv_off[k], ibt = invT_off[k];
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  const int64_t tsz = (int64_t)B * B;
  {
    // InvT(tq, tq) = Linv_tq^T
    const float2* src = Linv + (int64_t)(t0 + tq) * tsz + cs;
    float2* dst = InvT + (ibt + tq * (tq + 1) / 2 + tq) * tsz + (int64_t)cs * B;
    for (int i = threadIdx.x; i < B * CW; i += IT) sC[(i / CW) * LDC + i % CW] = src[(int64_t)(i / CW) * B + i % CW];
    __syncthreads();
    for (int i = threadIdx.x; i < B * CW; i += IT) dst[i] = sC[(i % B) * LDC + i / B];
    __syncthreads();
  }
  for (int t = tq + 1; t < nt; ++t) {
    float2 acc[TM][4];
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) acc[i][j] = make_float2(0.f, 0.f);
    // C = sum_s L(t, s) Inv(s, tq)
    for (int s = tq; s < t; ++s) {
      const float2* A = L + (tcolptr[t0 + s] + (t - s)) * tsz;
      const float2* Bm = (s == tq) ? Linv + (int64_t)(t0 + tq) * tsz : Inv + (ib + s * (s - 1) / 2 + tq) * tsz;
      gemm_strip<B, true>(A, Bm + cs, sA, sB, acc);
    }
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        sC[(ty * TM + i) * LDC + tx + 16 * j] = acc[i][j];
        acc[i][j] = make_float2(0.f, 0.f);
      }
    // Inv(t, tq) = -Linv_tt C (the product's first barrier orders C)
    gemm_strip<B, false>(Linv + (int64_t)(t0 + t) * tsz, sC, sA, sB, acc);
    float2* out = Inv + (ib + t * (t - 1) / 2 + tq) * tsz + cs;
    float2* outT = InvT + (ibt + t * (t + 1) / 2 + tq) * tsz + (int64_t)cs * B;
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        acc[i][j] = make_float2(-acc[i][j].x, -acc[i][j].y);
        out[(int64_t)(ty * TM + i) * B + tx + 16 * j] = acc[i][j];
      }
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int i = 0; i < TM; i += 2)
        *reinterpret_cast<float4*>(outT + (int64_t)(tx + 16 * j) * B + ty * TM + i) =
            make_float4(acc[i][j].x, acc[i][j].y, acc[i + 1][j].x, acc[i + 1][j].y);
    __syncthreads();   // Inv(t, tq) is read back by this block for the next t
  }
}

}  // namespace

int launch_inv_build(const int2* work, int nwork, const int32_t* tstart, const int64_t* tcolptr,
                     const int64_t* inv_off, const int64_t* invT_off, const void* L, const void* Linv, void* Inv,
                     void* InvT, int b, cudaStream_t st) {
  if (nwork <= 0) return 0;
  const size_t smem = sizeof(float2) * ((size_t)KC * (b + 2) + (size_t)KC * CW + (size_t)b * LDC);
  if (b == 128) {
    cudaFuncSetAttribute(inv_build_kernel<128>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    inv_build_kernel<128><<<nwork * (128 / CW), IT, smem, st>>>(work, tstart, tcolptr, inv_off, invT_off, (const float2*)L,
                                                   (const float2*)Linv, (float2*)Inv, (float2*)InvT);
  } else if (b == 64) {
    cudaFuncSetAttribute(inv_build_kernel<64>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    inv_build_kernel<64><<<nwork * (64 / CW), IT, smem, st>>>(work, tstart, tcolptr, inv_off, invT_off, (const float2*)L,
                                                  (const float2*)Linv, (float2*)Inv, (float2*)InvT);
  } else {
    return (int)cudaErrorInvalidValue;
  }
  return (int)cudaGetLastError();
}

}  // namespace d3m
