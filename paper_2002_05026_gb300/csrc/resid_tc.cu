// FP64-accurate residual r = b - K x on the tcgen05 tensor cores (the refinement's residual:
// FP64 on the GPU only for r = b - K x and the solution update).
//
// Method: an exact-product splitting in the manner of Ozaki, Ogita, Oishi and Rump ("Error-free
// transformations of matrix multiplication by using fast routines of matrix multiplication and
// its applications", Numer. Algorithms 2012), with the slices held as small integers in FP8 (e4m3):
//  * every stored block K_fg gets one scale 2^E (max |Re|, |Im| over the block < 2^E; the
//    diagonal entries of a diagonal block are left out of the block and applied in FP64); the
//    normalised entries k = K 2^-E are written as 11 balanced base-32 digits,
//        k ~ sum_{s=0..10} a_s 2^(-4 - 5 s),  a_0 in [-16, 16], a_s in [-16, 15] (s > 0),
//    each digit an integer that e4m3 holds exactly (|k - sum| <= 2^-55);
//  * every block of x (block g, right-hand side j) gets its own scale 2^T and digits b_q the
//    same way;
//  * a digit product a_s b_q is an integer of at most 256, so the tensor core's FP32
//    accumulation of all products of one level t = s + q over a block of up to 512 columns
//    (2 x 512 terms with the real embedding of the complex product, at most 11 digit pairs a
//    level) stays below 2^21.5 and is EXACT; the levels t = 0..11 (76 digit pairs) are kept, the
//    dropped ones sum to about 2^-55 of the scales' product;
//  * the twelve exact level sums of a block are combined exactly in two 64-bit integers, rounded
//    once to FP64 in integer arithmetic (conversions run at the FP64 rate), scaled by 2^(E + T)
//    and accumulated in FP64; r = b - acc - diag(K) x.
// Why e4m3: the kernel streams the digit planes and is bound by their bytes and by the tensor
// rate.  11 bytes an entry and orientation where nine base-64 digits in bf16 take 18, and 76 products at
// twice the bf16 rate where 45 are needed at the bf16 rate.  Measured per call: 5x5x4 blocks of 512, 32 right-hand
// sides, 6.4 -> 3.56 ms; 8x8 of 512, 8 of them, 1.13 -> 0.62 ms (nine bf16 digits before).  Without the
// products of A digits 2.. these take 2.40 and 0.60 ms: 8 right-hand sides are at the rate of the digit
// planes' bytes, 32 half-way between bytes and products.  The group width is a template argument: with
// descriptors formed at run time by the one issuing lane the MMAs ran at half this rate (5.75 ms).
// Complex products use the real embedding along K: A = [a_r | a_i] (row u, 2 x 32 columns per
// chunk), B = [[b_r, b_i]; [-b_i, b_r]] (N = 2 NR output columns: Re of NR right-hand sides,
// then Im).  The digit planes of B are stacked, and so are the levels in TMEM, so that one MMA
// (N' = min(11, 12 - a) N columns, split beyond 256) multiplies A digit a by every B digit it meets.
//
// Data (e4m3 digit planes of 128 or N rows x 32 columns = 32-byte rows, stored 32-byte swizzled as the
// MMA reads them, so that a stage is two contiguous bulk copies; a tensor-map copy of 32-byte rows ran at
// the rate of its rows): K digits per residual contribution (row tile, 32-column chunk, part r/i, digit), both
// orientations of an off-diagonal block stored (written once per factorization); x digits per
// block g (chunk, part, digit) and N rows (written per residual call).
//
// Kernel roles (320 threads): warp 0 issues the TMA loads (four 55 KB stages: 11 A planes of one
// part + 11 B planes), warp 1 issues the MMAs into 12 level accumulators in TMEM (12 x N <= 384
// columns, N = 2 NR <= 32: at most 16 right-hand sides a group; two sets of them for N = 16), warps
// 2..9 read the levels back after every block and accumulate.
#include <cuda_runtime.h>

#include "d3m.h"
#include "device.cuh"
#include "kernels.h"

namespace d3m {

namespace {

constexpr int RT_WARPS = 10;
constexpr int RT_THREADS = RT_WARPS * 32;
constexpr int ND = kResidDigits;                   // digits per value
constexpr int NL = ND + 1;                         // levels kept: 0..NL-1
constexpr int NRMAX = 16;                          // right-hand sides per group (N = 2 NR <= 32)
constexpr uint32_t APLANE = 128 * 32;              // 4 KB: 128 rows x 32 digits
constexpr uint32_t BPLANE = 32 * 32;               // 1 KB: at most 32 rows x 32 digits
constexpr uint32_t A_STAGE = ND * APLANE;          // 44 KB
constexpr uint32_t STG = A_STAGE + ND * BPLANE;    // 55 KB
constexpr int NSTG = 4;
constexpr uint32_t RT_SMEM = NSTG * STG;           // 220 KB
static_assert(STG % 1024 == 0 && NL * 2 * NRMAX <= 512, "stage layout / TMEM columns");
constexpr int UNIT_KC = 16;                        // 32-column chunks per accumulation unit (512 columns)

__device__ __forceinline__ uint32_t su32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void bar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void bar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void bar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ bool bar_try(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}
__device__ __forceinline__ bool bar_wait(uint32_t bar, uint32_t parity, uint64_t deadline) {
  while (!bar_try(bar, parity)) {
    if (globaltimer_ns() > deadline) return false;
  }
  return true;
}
// `bytes` contiguous bytes (16-byte aligned, a multiple of 16) into shared memory
__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst), "l"(src),
               "r"(bytes), "r"(bar)
               : "memory");
}
// 16-byte unit h of row r of a digit plane (32-byte rows): the planes lie in global memory as the MMA reads
// them from shared memory, 32-byte swizzled
__device__ __forceinline__ int swz_unit(int r, int h) { return r * 32 + ((h ^ ((r >> 2) & 1)) << 4); }
// K-major, 32-byte swizzle, 8-row groups 256 bytes apart
__device__ __forceinline__ uint64_t sdesc(uint32_t saddr) {
  uint64_t d = (uint64_t)((saddr & 0x3FFFFu) >> 4);
  d |= (uint64_t)1 << 16;
  d |= (uint64_t)(256u >> 4) << 32;
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)6 << 61;
  return d;
}
// kind::f8f6f4, A and B e4m3 (format 0), D f32, K-major, M = 128
__device__ __forceinline__ uint32_t idesc_f8(uint32_t n) { return (1u << 4) | ((n >> 3) << 17) | ((128u >> 4) << 24); }
__device__ __forceinline__ void mma_f8(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t accum) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f8f6f4 [%0], %1, %2, %3, p;\n}\n" ::"r"(d),
      "l"(a), "l"(b), "r"(idesc), "r"(accum)
      : "memory");
}
__device__ __forceinline__ void mma_commit_bar(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t* r) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];\n"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr));
}
// wait for the loads; each value then passes through a wait of its own, so that no use moves before it
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ float loaded(uint32_t r) {
  asm volatile("" : "+r"(r));
  return __uint_as_float(r);
}

// Fixed-point word of a double relative to the scale 2^E (|x| < 2^E): F = x 2^(54 - E) rounded to nearest,
// plus 16 in each of its ten low base-32 places, so that place s holds digit + 16 (and the bits above
// them the leading digit): x 2^-E ~ sum_s d[s] 2^(-4 - 5 s), d[0] in [-16, 16], d[s] in [-16, 15].
// Integer operations only.  Zeros, subnormals and values below 2^(E-55) give all-zero digits.
__device__ __forceinline__ long long digit_word(double x, int E) {
  const unsigned long long u = (unsigned long long)__double_as_longlong(x);
  const int be = (int)((u >> 52) & 0x7ff);
  long long F = 0;
  if (be != 0 && be != 0x7ff) {
    const unsigned long long mant = (u & 0xFFFFFFFFFFFFFull) | (1ull << 52);
    const int sh = be - 1021 - E;          // x 2^(54 - E) = mant 2^(be - 1075 + 54 - E)
    unsigned long long a;
    if (sh >= 0) a = mant << (sh > 1 ? 1 : sh);     // |x| < 2^E keeps sh <= 1 (|a| <= 2^54)
    else if (sh > -64) a = (mant + (1ull << (-sh - 1))) >> (-sh);
    else a = 0;
    F = (u >> 63) ? -(long long)a : (long long)a;
  }
  return F + 0x2108421084210ll;            // sum_{p < 10} 16 32^p
}
// digit s of a word plus 16, in [0, 32]
__device__ __forceinline__ int digit_at(long long w, int s) {
  const int v = (int)(w >> (50 - 5 * s));
  return s == 0 ? v + 16 : (v & 31);
}
// e4m3 code of an integer v, |v| <= 16
__device__ __forceinline__ unsigned char e4m3_of(int v) {
  const int m = v < 0 ? -v : v;
  const int c = m >= 8 ? 0x48 + m : (m >= 4 ? 0x40 + 2 * m : (m >= 2 ? 0x38 + 4 * m : (m ? 0x38 : 0)));
  return (unsigned char)(v < 0 ? c | 0x80 : c);
}

// |x| as its bits (ordered like the values, without FP64 compares; a NaN counts as 0)
__device__ __forceinline__ unsigned long long mag_bits(double x) {
  const unsigned long long u = (unsigned long long)__double_as_longlong(x) & 0x7fffffffffffffffull;
  return u > 0x7ff0000000000000ull ? 0ull : u;
}

// exponent E with |v| < 2^E for the largest magnitude v (as double bits); 0 for v = 0
__device__ __forceinline__ int scale_exp(unsigned long long maxbits) {
  const int be = (int)((maxbits >> 52) & 0x7ff);
  return be == 0 ? 0 : be - 1022;
}

// ---------------------------------------------------------------- K digits
// (1) per stored block (bound by HBM; a division by the block's height only where the diagonal lies in it, 8 x 8 of
// 512: 0.35 -> 0.28 ms): max |Re|, |Im| (diagonal entries of a diagonal block excluded) as double
// bits, and the diagonal entries of the diagonal blocks (applied in FP64 by the residual)
__global__ void __launch_bounds__(256) kblock_max_kernel(ResidualTc p) {
  const int blk = blockIdx.x;
  const int f = p.blk_row[blk], g = p.blk_col[blk];
  const int mf = p.m_orig[f], mg = p.m_orig[g];
  const double2* Kb = p.K + p.kblk_off[blk];
  const int64_t tot = (int64_t)mf * mg;
  unsigned long long mx = 0;
  const int64_t stride = 256 * gridDim.y;
  auto take = [&](double2 v) {
    const unsigned long long ab = (unsigned long long)__double_as_longlong(fmax(fabs(v.x), fabs(v.y)));
    mx = ab > mx ? ab : mx;
  };
  if (f != g) {
    int64_t i = blockIdx.y * 256 + threadIdx.x;
    for (; i + 3 * stride < tot; i += 4 * stride) {   // four loads in flight
      double2 v[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) v[e] = __ldg(Kb + i + e * stride);
#pragma unroll
      for (int e = 0; e < 4; ++e) take(v[e]);
    }
    for (; i < tot; i += stride) take(__ldg(Kb + i));
  } else {
    for (int64_t i = blockIdx.y * 256 + threadIdx.x; i < tot; i += stride) {
      const double2 v = __ldg(Kb + i);
      const int c = (int)(i / mf), u = (int)(i - (int64_t)c * mf);
      if (u == c) p.Kdiag[p.xoff_orig[f] + u] = v;
      else take(v);
    }
  }
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long t = __shfl_xor_sync(0xffffffffu, mx, o);
    mx = t > mx ? t : mx;
  }
  if ((threadIdx.x & 31) == 0 && mx) atomicMax(p.Kmax_bits + blk, mx);
}

// (2) digits of the stored blocks: one tile of 64 rows x 32 columns of a stored block K_fg (f >= g) per
// CTA (50 KB of shared memory: four CTAs per SM, so that the loads, digits and stores of different tiles overlap; 128
// rows and two CTAs took 1.66 ms for 8 x 8 blocks of 512 where this takes 1.27).  Every entry's 2 ND digits are extracted once, into
// shared memory (their e4m3 codes, [plane][row u][column c]), and written to the planes of both
// residual contributions of the block: row block f (untransposed: one 32-column chunk of 128 rows u) and, for
// f != g, row block g (transposed, by 4 x 4 byte transposes: 32 of the 128 rows c, four 32-column chunks of
// u).  K is read once, coalesced along u (column-major blocks).  Also adds |K| row sums (rows u) and column
// sums (rows c of the transposed use) into rowsum, for ||K||_inf.  Bound by HBM: 16 bytes read and 2 x 22
// written an entry.
constexpr int KD_U = 64, KD_C = 32, KD_LD = 36;     // tile rows, tile columns, padded bytes of a row
constexpr size_t KD_SMEM = (size_t)2 * ND * KD_U * KD_LD;

__global__ void __launch_bounds__(256) kdigits_kernel(ResidualTc p) {
  extern __shared__ __align__(16) unsigned char sdig[];   // [2 ND][KD_U][KD_LD]
  __shared__ float s_cs[KD_C];
  __shared__ unsigned char s_code[36];
  const int blk = blockIdx.x, rt = blockIdx.y, ct = blockIdx.z;
  const int f = p.blk_row[blk], g = p.blk_col[blk];
  const int mf = p.m_orig[f], mg = p.m_orig[g];
  if (rt * KD_U >= mf || ct * KD_C >= mg) return;   // the grid covers the largest blocks
  const int E = scale_exp(p.Kmax_bits[blk]);
  const double2* Kb = p.K + p.kblk_off[blk];
  const bool diag = (f == g);
  const int tid = threadIdx.x, lane = tid & 31, ul = tid % KD_U, ch = tid / KD_U;
  const int u = rt * KD_U + ul;
  if (tid < KD_C) s_cs[tid] = 0.f;
  if (tid < 33) s_code[tid] = e4m3_of(tid - 16);
  __syncthreads();
  float rs = 0.f;
#pragma unroll 1
  for (int q = 0; q < KD_C * KD_U / 1024; ++q) {
    // four columns c0 .. c0 + 3 of row u
    const int cl0 = ch * (KD_C * KD_U / 256) + q * 4;
    double2 v[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int c = ct * KD_C + cl0 + e;
      v[e] = (u < mf && c < mg) ? __ldg(Kb + (int64_t)c * mf + u) : make_double2(0.0, 0.0);
    }
    uint32_t dig[2 * ND];
#pragma unroll
    for (int s = 0; s < 2 * ND; ++s) dig[s] = 0;
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const float fx = (float)v[e].x, fy = (float)v[e].y;
      const float a = sqrtf(fx * fx + fy * fy);
      rs += a;
      float cs = a;
      for (int o = 16; o > 0; o >>= 1) cs += __shfl_xor_sync(0xffffffffu, cs, o);
      if (lane == 0) atomicAdd(&s_cs[cl0 + e], cs);
      if (diag && u == ct * KD_C + cl0 + e) v[e] = make_double2(0.0, 0.0);
      const long long wr = digit_word(v[e].x, E), wi = digit_word(v[e].y, E);
#pragma unroll
      for (int s = 0; s < ND; ++s) {
        dig[s] |= (uint32_t)s_code[digit_at(wr, s)] << (8 * e);
        dig[ND + s] |= (uint32_t)s_code[digit_at(wi, s)] << (8 * e);
      }
    }
#pragma unroll
    for (int s = 0; s < 2 * ND; ++s) *reinterpret_cast<uint32_t*>(sdig + (s * KD_U + ul) * KD_LD + cl0) = dig[s];
  }
  if (u < mf) atomicAdd(p.rowsum + p.xoff_orig[f] + u, rs);
  __syncthreads();
  if (!diag && tid < KD_C && ct * KD_C + tid < mg) atomicAdd(p.rowsum + p.xoff_orig[g] + ct * KD_C + tid, s_cs[tid]);
  // untransposed planes (row block f): chunk ct, whole 4 KB planes, 16-byte units
  {
    const int nkc = (mg + 31) / 32;
    unsigned char* base = p.kdig + ((int64_t)p.ks_plane[p.blk_eu[blk]] + ((int64_t)(rt / 2) * nkc + ct) * 2 * ND) * APLANE;
    const int r0 = (rt & 1) * KD_U;
    for (int w = tid; w < 2 * ND * KD_U * 2; w += 256) {
      const int h = w & 1, r = (w >> 1) % KD_U, pl = w / (2 * KD_U);
      const uint32_t* src = reinterpret_cast<const uint32_t*>(sdig + (pl * KD_U + r) * KD_LD + h * 16);
      *reinterpret_cast<uint4*>(base + pl * APLANE + swz_unit(r0 + r, h)) = make_uint4(src[0], src[1], src[2], src[3]);
    }
  }
  // transposed planes (row block g, source f): rows c, 32-column chunks of u; a unit is 16 u x 4 c
  if (!diag) {
    const int nkc = (mf + 31) / 32;
    unsigned char* base = p.kdig + ((int64_t)p.ks_plane[p.blk_et[blk]] + (int64_t)(ct / 4) * nkc * 2 * ND) * APLANE;
    const int r0 = (ct & 3) * KD_C;
    for (int w = tid; w < 2 * ND * KD_U / 2; w += 256) {
      const int h = w & 1, c4 = (w >> 1) & 7, kcl = (w >> 4) % (KD_U / 32), pl = w / (KD_U / 2);
      const int kc = rt * (KD_U / 32) + kcl;
      if (kc >= nkc) continue;
      const unsigned char* src = sdig + (pl * KD_U + kcl * 32 + h * 16) * KD_LD + c4 * 4;
      uint32_t o[4][4];                              // [c][4 u]
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        uint32_t x[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) x[k] = *reinterpret_cast<const uint32_t*>(src + (4 * i + k) * KD_LD);
        const uint32_t a = __byte_perm(x[0], x[1], 0x5140), b = __byte_perm(x[2], x[3], 0x5140);   // bytes 0, 1
        const uint32_t c = __byte_perm(x[0], x[1], 0x7362), d = __byte_perm(x[2], x[3], 0x7362);   // bytes 2, 3
        o[0][i] = __byte_perm(a, b, 0x5410);
        o[1][i] = __byte_perm(a, b, 0x7632);
        o[2][i] = __byte_perm(c, d, 0x5410);
        o[3][i] = __byte_perm(c, d, 0x7632);
      }
      unsigned char* dst = base + ((int64_t)kc * 2 * ND + pl) * APLANE + swz_unit(r0 + c4 * 4, h);   // the four rows swizzle alike
#pragma unroll
      for (int c = 0; c < 4; ++c) *reinterpret_cast<uint4*>(dst + c * 32) = make_uint4(o[c][0], o[c][1], o[c][2], o[c][3]);
    }
  }
}

// (3) ||K_i||_inf = max row sum over the rows of instance i
__global__ void rowsum_max_kernel(const float* __restrict__ rowsum, const int64_t* __restrict__ xoff_orig,
                                  const int32_t* __restrict__ m_orig, const int32_t* __restrict__ inst, int nblk,
                                  unsigned* kmax) {
  const int f = blockIdx.x;
  float mx = 0.f;
  for (int u = threadIdx.x; u < m_orig[f]; u += blockDim.x) mx = fmaxf(mx, rowsum[xoff_orig[f] + u]);
  for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  if ((threadIdx.x & 31) == 0) atomicMax(kmax + inst[f], __float_as_uint(mx));
}

// ---------------------------------------------------------------- x digits (per residual call)
// Block g, right-hand sides j0 .. j0 + NR - 1, chunks 4 z .. 4 z + 3: T_(g,j) from max |Re|, |Im| over the
// block's rows, then the B planes [chunk][part][digit] of N = 2 NR rows x 32 columns:
//   part r: row j -> b_r(c, j), row NR + j -> b_i(c, j);  part i: row j -> -b_i, row NR + j -> b_r.
constexpr int XD_KC = 4;                            // chunks per CTA
__global__ void __launch_bounds__(256) xdigits_kernel(ResidualTc p, const double2* __restrict__ X, int nrhs, int NR) {
  const int g = blockIdx.x, grp = blockIdx.y, j0 = grp * NR;
  if (p.done && p.done[p.inst[g]]) return;
  const int mg = p.m_orig[g];
  const int nkc = (mg + 31) / 32, k0 = blockIdx.z * XD_KC;
  if (k0 >= nkc) return;
  const int64_t xo = p.xoff_orig[g];
  __shared__ unsigned long long s_max[NRMAX];
  __shared__ int s_T[NRMAX];
  __shared__ unsigned char s_code[36];
  if (threadIdx.x < NRMAX) s_max[threadIdx.x] = 0;
  if (threadIdx.x < 33) s_code[threadIdx.x] = e4m3_of((int)threadIdx.x - 16);
  __syncthreads();
  // a warp takes 32 consecutive rows of one right-hand side at a time
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int jl = warp; jl < NR && j0 + jl < nrhs; jl += 8) {
    unsigned long long mx = 0;
    for (int c = lane; c < mg; c += 32) {
      const double2 v = X[(int64_t)(j0 + jl) * p.n + xo + c];
      mx = max(mx, max(mag_bits(v.x), mag_bits(v.y)));
    }
    for (int o = 16; o > 0; o >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if (lane == 0) s_max[jl] = mx;
  }
  __syncthreads();
  if (threadIdx.x < NR) {
    s_T[threadIdx.x] = scale_exp(s_max[threadIdx.x]);
    if (blockIdx.z == 0) p.xT[((int64_t)grp * p.nblk + g) * 32 + threadIdx.x] = s_T[threadIdx.x];
  }
  __syncthreads();
  const int k1 = min(nkc, k0 + XD_KC);
  const int bplane = 2 * NR * 32;                    // the planes of a call lie N rows apart
  unsigned char* planes = p.xdig + ((int64_t)grp * p.xs_total + p.xs_plane[g]) * bplane;
  // one thread per (chunk, right-hand side, 8 columns): digits of 8 entries, four rows of planes
  const int jobs = (k1 - k0) * NR * 4;
  for (int w = threadIdx.x; w < jobs; w += 256) {
    const int c8 = w & 3, j = (w >> 2) % NR, kc = k0 + (w >> 2) / NR;
    uint2 o[2][ND];                                  // [Re, Im][digit]
#pragma unroll
    for (int s = 0; s < ND; ++s) o[0][s] = o[1][s] = make_uint2(0u, 0u);
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const int c = kc * 32 + c8 * 8 + q;
      double2 v = make_double2(0.0, 0.0);
      if (c < mg && j0 + j < nrhs) v = X[(int64_t)(j0 + j) * p.n + xo + c];
      const long long wr = digit_word(v.x, s_T[j]), wi = digit_word(v.y, s_T[j]);
#pragma unroll
      for (int s = 0; s < ND; ++s) {
        const uint32_t dr = (uint32_t)s_code[digit_at(wr, s)] << (8 * (q & 3)), di = (uint32_t)s_code[digit_at(wi, s)] << (8 * (q & 3));
        if (q < 4) {
          o[0][s].x |= dr;
          o[1][s].x |= di;
        } else {
          o[0][s].y |= dr;
          o[1][s].y |= di;
        }
      }
    }
    // part r: Re rows take b_r, Im rows b_i; part i: Re rows take -b_i (sign bits), Im rows b_r
    unsigned char* pr = planes + (int64_t)kc * 2 * ND * bplane + (c8 & 1) * 8;
    unsigned char* pi = pr + ND * bplane;
    const int o1 = swz_unit(j, c8 >> 1), o2 = swz_unit(NR + j, c8 >> 1);
#pragma unroll
    for (int s = 0; s < ND; ++s) {
      *reinterpret_cast<uint2*>(pr + s * bplane + o1) = o[0][s];
      *reinterpret_cast<uint2*>(pr + s * bplane + o2) = o[1][s];
      *reinterpret_cast<uint2*>(pi + s * bplane + o1) = make_uint2(o[1][s].x ^ 0x80808080u, o[1][s].y ^ 0x80808080u);
      *reinterpret_cast<uint2*>(pi + s * bplane + o2) = o[0][s];
    }
  }
}

// ---------------------------------------------------------------- the residual kernel
template <int NR>   // right-hand sides per group: 8 or 16
__global__ void __launch_bounds__(RT_THREADS, 1)
    resid_tc_kernel(const ResidualTc p, const double2* __restrict__ X, const double2* __restrict__ B, double2* __restrict__ R, int nrhs, int ngrp) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* smem = smem_raw + ((1024u - (su32(smem_raw) & 1023u)) & 1023u);
  __shared__ __align__(8) uint64_t bar_full[NSTG], bar_empty[NSTG], bar_accf[2], bar_acce[2];
  __shared__ uint32_t s_tmem;
  __shared__ int s_fail;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  // the right-hand-side groups of one row tile are adjacent block indices, so they run together
  // and read the tile's K digits from L2 after the first one brought them in
  const int grp = blockIdx.x % ngrp, j0 = grp * NR;
  const int2 rtile = p.rtiles[blockIdx.x / ngrp];
  const int f = rtile.x, rt = rtile.y;
  if (p.done && p.done[p.inst[f]]) return;       // converged instance: r and its norms are kept
  const int mf = p.m_orig[f];
  constexpr int N = 2 * NR;
  const int64_t e0 = p.res_ptr[f], e1 = p.res_ptr[f + 1];
  const uint64_t deadline = globaltimer_ns() + (uint64_t)p.timeout_ns;

  if (tid == 0) {
    for (int s = 0; s < NSTG; ++s) {
      bar_init(su32(&bar_full[s]), 1);
      bar_init(su32(&bar_empty[s]), 1);
    }
    for (int s = 0; s < 2; ++s) {
      bar_init(su32(&bar_accf[s]), 1);
      bar_init(su32(&bar_acce[s]), RT_WARPS - 2);
    }
    s_fail = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(su32(&s_tmem)), "r"(512u)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = s_tmem;
  constexpr uint32_t bbytes = (uint32_t)N * 32;          // one B digit plane (N rows x 32 bytes)
  // sets of level accumulators: two (a block's products run while the one before is read back) if they fit
  constexpr uint32_t nset = 2 * NL * N <= 512 ? 2u : 1u;

  if (warp == 0) {
    // ------------------------------------------------------------ TMA producer
    if (lane == 0) {
      uint32_t it = 0;
      bool ok = true;
      for (int64_t e = e0; e < e1 && ok; ++e) {
        const int g = p.res_src[e];
        const int nkc = (p.m_orig[g] + 31) / 32;
        const int64_t abase = p.ks_plane[e] + (int64_t)rt * nkc * 2 * ND;
        const int64_t bbase = (int64_t)grp * p.xs_total + p.xs_plane[g];
        for (int kc = 0; kc < nkc && ok; ++kc)
          for (int part = 0; part < 2; ++part, ++it) {
            const uint32_t s = it % NSTG, use = it / NSTG;
            if (!bar_wait(su32(&bar_empty[s]), (use & 1) ^ 1, deadline)) { ok = false; break; }
            const uint32_t fb = su32(&bar_full[s]);
            bar_expect_tx(fb, A_STAGE + ND * bbytes);
            const uint32_t sa = su32(smem + s * STG);
            bulk_load(sa, p.kdig + (abase + (int64_t)(kc * 2 + part) * ND) * APLANE, A_STAGE, fb);
            bulk_load(sa + A_STAGE, p.xdig + (bbase + (int64_t)(kc * 2 + part) * ND) * bbytes, ND * bbytes, fb);
          }
      }
      if (!ok) atomicExch(&s_fail, 1);
    }
    __syncwarp();
  } else if (warp == 1) {
    // ------------------------------------------------------------ MMA issuer
    if (lane == 0) {
      uint32_t it = 0, unit = 0;
      bool ok = true;
      for (int64_t e = e0; e < e1 && ok; ++e) {
        const int g = p.res_src[e];
        const int nkc = (p.m_orig[g] + 31) / 32;
        for (int k0 = 0; k0 < nkc && ok; k0 += UNIT_KC, ++unit) {
          // the epilogue has read this set's previous levels
          const uint32_t set = unit % nset, suse = unit / nset;
          if (!bar_wait(su32(&bar_acce[set]), (suse & 1) ^ 1, deadline)) { ok = false; break; }
          fence_after();
          const uint32_t acc0 = tmem + set * (uint32_t)(NL * N);
          const int k1 = min(nkc, k0 + UNIT_KC);
          for (int kc = k0; kc < k1 && ok; ++kc)
            for (int part = 0; part < 2; ++part, ++it) {
              const uint32_t s = it % NSTG, use = it / NSTG;
              if (!bar_wait(su32(&bar_full[s]), use & 1, deadline)) { ok = false; break; }
              fence_after();
              const uint32_t sa = su32(smem + s * STG), sb = sa + A_STAGE;
              const bool first = (kc == k0 && part == 0);
              // A digit da meets B digits 0 .. min(ND, NL - da) - 1: those B planes are consecutive rows in
              // shared memory and their levels da .. consecutive TMEM columns, so one MMA covers all of
              // them (two of equal size beyond 256 columns).  Digit 0 of A opens levels 0 .. NL - 2 of this
              // unit (at its first stage), digit 1 the last level.
              const uint64_t db = sdesc(sb);
#pragma unroll
              for (int da = 0; da < ND; ++da) {
                const int cnt = ND < NL - da ? ND : NL - da;
                const uint64_t ad = sdesc(sa + da * APLANE);
                auto span = [&](int q0, int q1, uint32_t acc) {   // B digits q0 .. q1 - 1
                  mma_f8(acc0 + (uint32_t)((da + q0) * N), ad, db + (uint32_t)(q0 * N * 32 >> 4), idesc_f8((uint32_t)((q1 - q0) * N)), acc);
                };
                const uint32_t acc = first && da == 0 ? 0u : 1u;
                if (da == 1 && first) {
                  span(0, 5, 1u);
                  span(5, ND - 1, 1u);
                  span(ND - 1, ND, 0u);
                } else if (cnt * N > 256) {
                  span(0, cnt / 2, acc);
                  span(cnt / 2, cnt, acc);
                } else {
                  span(0, cnt, acc);
                }
              }
              mma_commit_bar(su32(&bar_empty[s]));
            }
          mma_commit_bar(su32(&bar_accf[set]));
        }
      }
      if (!ok) atomicExch(&s_fail, 1);
    }
    __syncwarp();
  } else {
    // ------------------------------------------------------------ epilogue (8 warps)
    const int quad = warp & 3, hpart = (warp - 2) >> 2;   // TMEM lanes 32 quad.., Re (0) / Im (1)
    const int row = quad * 32 + lane;
    const int u = rt * 128 + row;
    double acc[NR];
#pragma unroll
    for (int j = 0; j < NR; ++j) acc[j] = 0.0;
    uint32_t unit = 0;
    bool ok = true;
    for (int64_t e = e0; e < e1 && ok; ++e) {
      const int g = p.res_src[e];
      const int nkc = (p.m_orig[g] + 31) / 32;
      const int E = scale_exp(p.Kmax_bits[p.res_blk[e]]);
      const int* Tg = p.xT + ((int64_t)grp * p.nblk + g) * 32;
      for (int k0 = 0; k0 < nkc; k0 += UNIT_KC, ++unit) {
        const uint32_t set = unit % nset, suse = unit / nset;
        if (!bar_wait(su32(&bar_accf[set]), suse & 1, deadline)) { ok = false; break; }
        fence_after();
        const uint32_t t0 = tmem + ((uint32_t)(quad * 32) << 16) + set * (uint32_t)(NL * N) + (uint32_t)(hpart * NR);
#pragma unroll
        for (int jb = 0; jb < NR; jb += 8) {
          {
            // the level sums are exact integers below 2^22 (to int by a magic-number add: a conversion takes
            // eight cycles a warp): levels 0..5 and 6..11 are combined exactly in 64-bit integers
            uint32_t v[NL][8];
#pragma unroll
            for (int t = 0; t < NL; ++t) tmem_ld8(t0 + (uint32_t)(t * N + jb), v[t]);
            tmem_wait_ld();
#pragma unroll
            for (int q = 0; q < 8; ++q) {
              int l[NL];
#pragma unroll
              for (int t = 0; t < NL; ++t) l[t] = __float_as_int(loaded(v[t][q]) + 12582912.f) - 0x4B400000;
              const long long u1 = (long long)((l[0] * 32 + l[1]) * 32 + l[2]) * 32768 + ((l[3] * 32 + l[4]) * 32 + l[5]);
              const long long u2 = (long long)((l[6] * 32 + l[7]) * 32 + l[8]) * 32768 + ((long long)l[9] * 1024 + (l[10] * 32 + l[11]));
              // value = (u1 2^-33 + u2 2^-63) 2^(E + T): level t weighs 2^(-8 - 5 t)
              int ex = E + Tg[jb + q];
              ex = ex < -900 ? -900 : (ex > 900 ? 900 : ex);
              acc[jb + q] += fixed_to_double<30>(u1, u2, ex - 63);
            }
          }
        }
        fence_before();
        __syncwarp();
        if (lane == 0) bar_arrive(su32(&bar_acce[set]));
      }
    }
    if (!ok) atomicExch(&s_fail, 1);
    // r = b - acc - diag(K) x in FP64, and the maxima for omega
    const bool active = ok && u < mf;
    const int64_t xo = p.xoff_orig[f];
    const double2 kd = active ? p.Kdiag[xo + u] : make_double2(0.0, 0.0);
#pragma unroll
    for (int q = 0; q < NR; ++q) {
      const int j = j0 + q;
      if (active && j < nrhs) {
        const int64_t o = (int64_t)j * p.n + xo + u;
        const double2 xv = X[o], bv = B[o];
        // this thread holds one part (Re or Im) of the block sums; the two parts of row u are
        // written by the two warps that share its TMEM lane quadrant
        if (hpart == 0) {
          const double dx = kd.x * xv.x - kd.y * xv.y;
          R[o].x = bv.x - acc[q] - dx;
        } else {
          const double dx = kd.x * xv.y + kd.y * xv.x;
          R[o].y = bv.y - acc[q] - dx;
        }
      }
    }
    // both parts are written: the norms are taken by the Re warps after a barrier among the
    // epilogue warps (named barrier 1, 256 threads)
    asm volatile("bar.sync 1, 256;" ::: "memory");
    if (hpart == 0) {
#pragma unroll 1
      for (int q = 0; q < NR; ++q) {
        const int j = j0 + q;
        float a = 0.f, x = 0.f, b = 0.f;
        if (active && j < nrhs) {
          const int64_t o = (int64_t)j * p.n + xo + u;
          const double2 r = R[o], xv = X[o], bv = B[o];
          const float rx = (float)r.x, ry = (float)r.y;
          a = sqrtf(rx * rx + ry * ry);
          const float xx = (float)xv.x, xy = (float)xv.y;
          x = sqrtf(xx * xx + xy * xy);
          const float bx = (float)bv.x, by = (float)bv.y;
          b = sqrtf(bx * bx + by * by);
        }
        for (int o = 16; o > 0; o >>= 1) {
          a = fmaxf(a, __shfl_xor_sync(0xffffffffu, a, o));
          x = fmaxf(x, __shfl_xor_sync(0xffffffffu, x, o));
          b = fmaxf(b, __shfl_xor_sync(0xffffffffu, b, o));
        }
        if (lane == 0 && j < nrhs) {
          const int qq = p.inst[f] * p.ld_norm + j0 + q;
          atomicMax(p.rmax + qq, __float_as_uint(a));
          atomicMax(p.xmax + qq, __float_as_uint(x));
          atomicMax(p.bmax + qq, __float_as_uint(b));
        }
      }
    }
  }

  __syncthreads();
  if (s_fail) {
    if (tid == 0) atomicExch(p.status, D3M_ERR_TIMEOUT);
    // give in-flight copies and MMAs time to land (bounded) before the memory is released
    const uint64_t t0 = globaltimer_ns();
    while (globaltimer_ns() - t0 < 2000000ull) __nanosleep(1000);
  }
  fence_before();
  __syncthreads();
  fence_after();
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u) : "memory");
}

}  // namespace

// digits of K (once per factorization, on the given stream), and ||K_i||_inf
int launch_kdigits(const ResidualTc& p, int nnzb, int nres, int max_rtiles, int nblk, cudaStream_t st) {
  cudaMemsetAsync(p.Kmax_bits, 0, (size_t)nnzb * sizeof(unsigned long long), st);
  cudaMemsetAsync(p.rowsum, 0, (size_t)p.n * sizeof(float), st);
  kblock_max_kernel<<<dim3((unsigned)nnzb, 8), 256, 0, st>>>(p);
  cudaFuncSetAttribute(kdigits_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)KD_SMEM);
  kdigits_kernel<<<dim3((unsigned)nnzb, (unsigned)(max_rtiles * (128 / KD_U)), (unsigned)(4 * max_rtiles)), 256, KD_SMEM, st>>>(p);
  rowsum_max_kernel<<<nblk, 128, 0, st>>>(p.rowsum, p.xoff_orig, p.m_orig, p.inst, nblk, p.kmax);
  return (int)cudaGetLastError();
}

// number of right-hand-side groups of one residual and their width NR (8 or 16)
int resid_tc_groups(int nrhs, int* NR) {
  const int ng = (nrhs + NRMAX - 1) / NRMAX;
  const int per = (nrhs + ng - 1) / ng;
  *NR = (per + 7) / 8 * 8;
  return ng;
}

// r = b - K x for the right-hand sides [0, nrhs): the digits of x for every group, then one launch
// with the groups of a row tile as adjacent blocks
int launch_resid_tc(const ResidualTc& p, const double2* X, const double2* B, double2* R,
                    int nrhs, int nrtiles, int nblk, int max_rtiles, cudaStream_t st, int64_t* launches) {
  const size_t smem = RT_SMEM + 1024;
  int NR = 8;
  const int ng = resid_tc_groups(nrhs, &NR);
  auto* kernel = NR == 8 ? resid_tc_kernel<8> : resid_tc_kernel<16>;
  cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return (int)e;
  xdigits_kernel<<<dim3((unsigned)nblk, (unsigned)ng, (unsigned)((4 * max_rtiles + XD_KC - 1) / XD_KC)), 256, 0, st>>>(p, X, nrhs, NR);
  kernel<<<(unsigned)(nrtiles * ng), RT_THREADS, smem, st>>>(p, X, B, R, nrhs, ng);
  *launches += 2;
  return (int)cudaGetLastError();
}

}  // namespace d3m
