// Persistent block-DAG factorization in FP64 with the tile products on the tensor cores (tile
// edge 64, complex128 factors): the D3M_FP64 engine.
//
// GB300 issues two FP64 FMAs per clock and SM, so one 64 x 64 x 64 complex tile product is 1.05 M
// DFMA = 0.25 ms of an SM, and both a task graph's throughput and its critical path are bound by
// that pipe.  Here every product of the factorization (the Schur updates S_IJ -= L_IK W_JK^T,
// W = L D, and the triangular solve W_IJ = S_IJ X_JJ^T, X = L_JJ^{-1}) is an exact integer product
// on tcgen05, in the manner of Ozaki, Ogita, Oishi and Rump ("Error-free transformations of matrix
// multiplication by using fast routines of matrix multiplication and its applications", Numer.
// Algorithms 2012):
//  * every row of an operand tile has a scale 2^E above its largest |Re|, |Im| (after a power-of-two
//    balance of the columns, see balance_of); an entry is held
//    as the 56-bit integer F = x 2^(54 - E) rounded to nearest (|error| <= 2^-55 of the scale; subnormals as zero),
//    biased by 0x80 in each of its seven bytes, so byte s of the word is 128 + the balanced base-256 digit
//    d_s in [-128, 127].  A finished tile is stored in this form beside its complex128 values;
//  * a digit is an exact bf16.  One tensor-core level t sums the digit products d_s d_q, s + q = t,
//    over the tile's 64 complex columns (128 terms of the real embedding, at most 7 pairs): an
//    integer below 7 * 128 * 2^14 < 2^24, exact in the FP32 accumulator.  Levels 0..7 are kept (34
//    digit pairs); the dropped ones sum to about 2^-59 of the scales' product (level 7 alone to 2^-51);
//  * the level sums of a tile product are combined exactly in 64-bit integers and added, aligned
//    by their scales, to a 128-bit fixed-point sum per output (two 64-bit words) over all products
//    of the task: a task rounds to FP64 once, at its end.
// The error of one product is about sqrt(128) 2^-54.8 of the product of the two rows' largest entries, that of FMAs
// a part 2^-53 of the terms' sum.  So an output of the digits falls short of FP64 where the two rows are large in
// different columns: unknowns in groups that couple weakly, a coupling that decays, anything but a diagonal scaling,
// which the balance removes.  Every row therefore carries its near columns, those within 2^-2 of its largest
// exponent.  Two rows that share one have sum |a_k b_k| >= 2^-6 of the scales' product; an output whose rows share
// none (or whose scales lie 2^13 below those of the task's largest product, or near the subnormal numbers, or in
// rows with an Inf or NaN) is formed by FP64 FMAs (fma_outputs), unless its rows meet in zeros only, which the
// nonzero columns of a row tell: two uncoupled groups of unknowns 24 ms instead of 253.  X_JJ and a panel's X_kk are held without their
// unit diagonal, whose term is added in FP64: it would set the scale of every row of a dominant tile; beside it a
// product may be short if 2^SLACK of the term reaches the scales'.  Error of the worst of the groups of unknowns of a
// dense system, coupled by eps^|g_i - g_j| and driven in one of them, largest of three draws (digits alone, digits
// and FMAs, FMAs alone): two groups, eps = 1e-4: 1.7e-12, 4.1e-16, 7.9e-16; 1e-8: 1.7e-8, 3.6e-16, 6.2e-16; eight groups, eps
// = 2^-4: 2.4e-8, 4.9e-16, 7.4e-16 (SLACK = 6: 2.1e-15; with pivoting 6.2e-16 and 6.2e-16); eps = 1 / 2: - , 5.2e-16,
// 7.6e-16; no groups: 4.9e-16, 4.1e-16, 7.1e-16.
// Cost, 4 x 4 grid, m = 512: dense: 2 % of the tasks have a few such outputs, factorization 20.2 -> 21.4 ms (an update
// of eight products 104 -> 106 us, an off-diagonal tile 44 -> 52, a diagonal one 162 -> 172); two and eight groups:
// 250 and 310 ms (FMAs alone: 255).
//
// One product: MMA M = 128 rows [Re c | Im c] of the embedded W (rows [b_r | -b_i], then
// [b_i | b_r]), N up to 448 = digits x 64 rows of L ([a_r | a_i]), K = 16 complex columns a
// stage; digit s of W meets digits 0 .. min(6, 7 - s) of L, which are consecutive rows, and fills
// consecutive level columns of TMEM.  2,176 tensor cycles a stage, 4 stages a product.
// All 16 warps expand the digits of a stage (8 words and 7 or 14 16-byte stores a thread) and read
// the levels back; a thread of the last warp also issues the MMAs (a seventeenth warp would cost
// every thread a quarter of its registers).  The expansion of the next stages overlaps the MMAs, the read-back
// does not (8 levels x 64 columns fill the tensor memory).
//
// Measured on GB300, factorization of a 4 x 4 grid with m = 512 (127 k products): 255 ms with DFMA tile
// products (1.04 TFLOP/s, 83 % of the FP64 pipe), 21 ms here; 3 x 3 grid with m = 100: 12.3 -> 3.0 ms.  A
// product takes about 20 k cycles (DFMA: 524 k), 8.7 k of them MMAs: two stages do not hide the
// expansion (2 k a stage) behind them, and the read-back (6 k) waits for the last one.  A diagonal tile
// takes about 170 us with the update before it (22 us), 16 us of it per 16-column pivot chain.  Solutions against 64-bit references: as far off as with DFMA
// (1.4e-15 and 1.1e-15 for these two).
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "device.cuh"
#include "diag_bk.cuh"
#include "kernels.h"

namespace d3m {

namespace {

constexpr int TB = 64;
constexpr int NWK = 16;                          // warps
constexpr int NTHR = NWK * 32;
constexpr int ISSUER = NWK - 1;                  // an L-side warp: its expansion has half the stores
constexpr int NDG = 7;                           // digits of an entry
constexpr int NLV = 8;                           // levels kept
constexpr uint32_t MPLANE = 128 * 64;            // one digit of 128 embedded W rows, 64-byte rows
constexpr uint32_t NPLANE = TB * 64;             // one digit of 64 L rows
constexpr uint32_t STAGE_N = NDG * MPLANE;       // offset of the L digits in a stage
constexpr uint32_t STAGE = NDG * (MPLANE + NPLANE);
constexpr int NSTG = 2;
constexpr uint32_t SMEM_BYTES = NSTG * STAGE;    // 168 KB
constexpr int LDS = 65;                          // c128 row stride of a tile in shared memory
constexpr int CH = 16;                           // complex columns of a stage
constexpr int NCH = TB / CH;
constexpr int MAXP = kDigMaxProducts;            // products of one task
constexpr int PW = CH;                           // panel width of a diagonal tile
constexpr uint32_t SMEM_S = STAGE;               // the tile of a diagonal task, behind one stage
static_assert(STAGE + TB * LDS * 16 + 2 * TB * (PW + 1) * 8 <= SMEM_BYTES, "shared memory of a diagonal task");
constexpr uint32_t OLD_OFF = 64 * 1024;          // exponents of S in a triangular solve: short2 [TB][TB]
constexpr unsigned long long BIAS = 0x0080808080808080ull;
constexpr int E_BAD = 8192;                      // scale of a row with an Inf or NaN
static_assert(TB * LDS * 16 <= SMEM_BYTES && STAGE % 1024 == 0, "shared memory");

__device__ __forceinline__ uint32_t su(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void bar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void bar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ bool bar_wait(uint32_t bar, uint32_t parity, uint64_t deadline) {
  for (;;) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    if (ok) return true;
    if (globaltimer_ns() > deadline) return false;
  }
}
// K-major, 64-byte swizzle, 8-row groups 512 bytes apart
__device__ __forceinline__ uint64_t sdesc(uint32_t saddr) {
  uint64_t d = (uint64_t)((saddr & 0x3FFFFu) >> 4);
  d |= (uint64_t)1 << 16;
  d |= (uint64_t)(512u >> 4) << 32;
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)4 << 61;
  return d;
}
__device__ __forceinline__ uint32_t idesc_bf16(uint32_t n) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((n >> 3) << 17) | ((128u >> 4) << 24);
}
__device__ __forceinline__ void mma_bf16(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t accum) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d),
      "l"(a), "l"(b), "r"(idesc), "r"(accum)
      : "memory");
}
__device__ __forceinline__ void mma_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tmem_ld2(uint32_t taddr, uint32_t* r) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x2.b32 {%0, %1}, [%2];\n" : "=r"(r[0]), "=r"(r[1]) : "r"(taddr));
}
// wait for the loads of v (tied to them, so that no use can move before the wait)
__device__ __forceinline__ void tmem_wait_ld(uint32_t (&v)[8][2]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+r"(v[0][0]), "+r"(v[0][1]), "+r"(v[1][0]), "+r"(v[1][1]), "+r"(v[2][0]), "+r"(v[2][1]), "+r"(v[3][0]),
                 "+r"(v[3][1]), "+r"(v[4][0]), "+r"(v[4][1]), "+r"(v[5][0]), "+r"(v[5][1]), "+r"(v[6][0]), "+r"(v[6][1]), "+r"(v[7][0]), "+r"(v[7][1])
               :
               : "memory");
}

// ------------------------------------------------------------------ words and digits
// exponent of x 2^shift as a biased double exponent (zero and subnormals: below every other; Inf and
// NaN: above)
constexpr int X_ZERO = -30000, X_BAD = 20000;
__device__ __forceinline__ int exp_of(double x, int shift) {
  const int be = (int)((__double_as_longlong(x) >> 52) & 0x7ff);
  return be == 0 ? X_ZERO : (be == 0x7ff ? X_BAD : be + shift);
}
// Row of an operand tile: its scale exponent from the largest exp_of its entries (that of a row of zeros is below
// every other), and its near columns, within 2^-NEAR of its largest entry (bit k: column k): all for a row of zeros,
// none with an Inf or NaN, or where a product with it may be subnormal
constexpr int E_ZERO = -3000, E_TINY = -450;
constexpr int NEAR = 2;
__device__ __forceinline__ int row_scale(int be) { return be >= X_BAD ? E_BAD : max(be - 1022, E_ZERO); }
__device__ __forceinline__ bool near_max(int e, int rowmax) { return e >= rowmax - NEAR; }
__device__ __forceinline__ bool no_near(int E) { return E >= E_BAD || (E < E_TINY && E > E_ZERO); }
// its nonzero columns; all for a row of zeros or with an Inf or NaN, so that the two meet
__device__ __forceinline__ uint2 row_nonzero(int rowmax, unsigned lo, unsigned hi) {
  return rowmax <= X_ZERO || rowmax >= X_BAD ? make_uint2(~0u, ~0u) : make_uint2(lo, hi);
}
__device__ __forceinline__ int4 row_info(int rowmax, unsigned lo, unsigned hi) {
  const int E = row_scale(rowmax);
  return no_near(E) ? make_int4(E, 0, 0, 0) : make_int4(E, 0, (int)lo, (int)hi);
}
constexpr int SLACK = 3;                         // see the top
constexpr int SPREAD = 13;                       // bits of the fixed-point sum past a product's own
constexpr int E_NONE = -100000;
// biased word of x 2^shift for scale 2^E (|x 2^shift| < 2^E): bytes 6..0 = digits 0..6 plus 128
__device__ __forceinline__ unsigned long long word_of(double x, int shift, int E) {
  const unsigned long long u = (unsigned long long)__double_as_longlong(x);
  const int be = (int)((u >> 52) & 0x7ff);
  unsigned long long a = 0;
  if (be != 0 && be != 0x7ff) {
    const unsigned long long mant = (u & 0xFFFFFFFFFFFFFull) | (1ull << 52);
    const int sh = be + shift - 1021 - E;         // x 2^(shift + 54 - E) = mant 2^sh, sh <= 1
    if (sh >= 0) a = mant << (sh > 1 ? 1 : sh);
    else if (sh > -64) a = (mant + (1ull << (-sh - 1))) >> (-sh);
  }
  return ((u >> 63) ? 0ull - a : a) + BIAS;
}
// balance of a column with pivot d: half its binary exponent.  Operands L and X = L^{-1} are held
// times 2^e per column, W = L D and S times 2^-e, so that a diagonal scaling of the matrix, which
// multiplies L[r][k] by s_r / s_k, leaves every row of an operand with one scale
__device__ __forceinline__ int balance_of(double2 d) {
  const int m = max(exp_of(d.x, 0), exp_of(d.y, 0));
  return (m <= X_ZERO || m >= X_BAD) ? 0 : (m - 1023) >> 1;
}
// the same for a column of a 2 x 2 pivot block (or three times the same pivot)
__device__ __forceinline__ int pair_balance(double2 d1, double2 d2, double2 e) {
  const int m = max(max(max(exp_of(d1.x, 0), exp_of(d1.y, 0)), max(exp_of(d2.x, 0), exp_of(d2.y, 0))),
                    max(exp_of(e.x, 0), exp_of(e.y, 0)));
  return (m <= X_ZERO || m >= X_BAD) ? 0 : (m - 1023) >> 1;
}
// digits of byte `sel` of two words (lo or hi halves x, y) as packed bf16: 128 + low 7 bits minus
// 128 or 256 by the byte's top bit, exact
__device__ __forceinline__ uint32_t digit_pair(uint32_t x, uint32_t y, uint32_t sel) {
  const uint32_t v = __byte_perm(x, y, sel);
  const uint32_t m = (v & 0x007f007fu) | 0x43004300u;
  const uint32_t c = (v & 0x00800080u) ^ 0x43804380u;
  const __nv_bfloat162 d = __hsub2(*reinterpret_cast<const __nv_bfloat162*>(&m), *reinterpret_cast<const __nv_bfloat162*>(&c));
  return *reinterpret_cast<const uint32_t*>(&d);
}
// word index of entry (row, k, part) of a tile: stages of 16 columns, [stage][row][part][16]
__device__ __forceinline__ int word_at(int row, int k, int part) { return (((k >> 4) * TB + row) * 2 + part) * CH + (k & 15); }

struct Words8 {
  ulonglong2 w[4];
};
__device__ __forceinline__ Words8 load_words(const unsigned long long* p) {
  Words8 r;
#pragma unroll
  for (int i = 0; i < 4; ++i) r.w[i] = __ldcg(reinterpret_cast<const ulonglong2*>(p) + i);
  return r;
}
// seven 16-byte units (8 bf16 digits each), digit s in out[s]
__device__ __forceinline__ uint4 digits8(const Words8& r, int s) {
  // digit s sits in byte 6 - s: digits 0..2 in the high half, 3..6 in the low half
  const bool hi = s < 3;
  const uint32_t byte = (uint32_t)(hi ? 2 - s : 6 - s);
  const uint32_t sel = byte | (byte << 4) | ((4u + byte) << 8) | ((4u + byte) << 12);
  uint32_t o[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const uint32_t x = hi ? (uint32_t)(r.w[i].x >> 32) : (uint32_t)r.w[i].x;
    const uint32_t y = hi ? (uint32_t)(r.w[i].y >> 32) : (uint32_t)r.w[i].y;
    o[i] = digit_pair(x, y, sel);
  }
  return make_uint4(o[0], o[1], o[2], o[3]);
}
__device__ __forceinline__ uint32_t unit_off(int row, int unit) {
  return (uint32_t)row * 64u + ((uint32_t)(unit ^ ((row >> 1) & 3)) << 4);
}

// the MMAs of one stage: digit d of W meets digits 0 .. min(6, 7 - d) of NR rows of L; level t takes
// the TMEM columns t NR ..
template <int NR>
__device__ __forceinline__ void stage_mmas(uint32_t tmem, uint32_t sm, bool open) {
  const uint64_t dm = sdesc(sm), dn = sdesc(sm + STAGE_N);   // offsets add to the descriptors' address field
#pragma unroll
  for (int kk = 0; kk < 2; ++kk)
#pragma unroll
    for (int d = 0; d < NDG; ++d) {
      // digit 0 opens levels 0..6 of a product, digit 1 level 7
      const bool first = open && kk == 0;
      const int cols = (d == 0 ? NDG : NLV - d) * NR;
#pragma unroll
      for (int off = 0; off < cols;) {
        int nn = cols - off < 256 ? cols - off : 256;
        if (d == 1 && off < 6 * NR && off + nn > 6 * NR) nn = 6 * NR - off;
        const uint32_t acc = first && (d == 0 || (d == 1 && off == 6 * NR)) ? 0u : 1u;
        mma_bf16(tmem + (uint32_t)(d * NR + off), dm + ((d * MPLANE + kk * 32) >> 4), dn + ((uint32_t)(off * 64 + kk * 32) >> 4),
                 idesc_bf16((uint32_t)nn), acc);
        off += nn;
      }
    }
}
// the digits of 8 entries (columns 8 k8 .. of a stage, part, row) into the stage's W or L planes
// (LROWS rows of L a stage)
template <int LROWS = TB>
__device__ __forceinline__ void put_digits(unsigned char* st, bool w_side, int row, int part, int k8, const Words8& w) {
  if (w_side) {
    // part r: b_r into rows c (first half) and 64 + c (second half); part i: -b_i into rows c
    // (second half), b_i into rows 64 + c (first half)
    const uint32_t o1 = unit_off(row, part * 2 + k8), o2 = unit_off(64 + row, (part ^ 1) * 2 + k8);
    const uint32_t neg = part ? 0x80008000u : 0u;
#pragma unroll
    for (int d = 0; d < NDG; ++d) {
      const uint4 v = digits8(w, d);
      *reinterpret_cast<uint4*>(st + d * MPLANE + o2) = v;
      *reinterpret_cast<uint4*>(st + d * MPLANE + o1) = make_uint4(v.x ^ neg, v.y ^ neg, v.z ^ neg, v.w ^ neg);
    }
  } else {
    const uint32_t o = unit_off(row, part * 2 + k8);
#pragma unroll
    for (int d = 0; d < NDG; ++d) *reinterpret_cast<uint4*>(st + STAGE_N + d * LROWS * 64 + o) = digits8(w, d);
  }
}

// x 2^k by its exponent field (zero and what leaves the range of normal numbers: 0)
__device__ __forceinline__ double scale2(double x, int k) {
  const long long u = __double_as_longlong(x);
  const int be = (int)((u >> 52) & 0x7ff) + k;
  return (((u >> 52) & 0x7ff) == 0 || be <= 0 || be >= 0x7ff) ? 0.0 : __longlong_as_double(u + ((long long)k << 52));
}
__device__ __forceinline__ double shfl_d(double v, int o) { return __shfl_xor_sync(0xffffffffu, v, o); }
// conversions between FP64 and FP32 by the bits (the conversion instructions run at the FP64 rate):
// to FP32 by truncation, for |x| in FP32's normal range (smaller: 0); to FP64 exactly, zero and
// normal numbers
__device__ __forceinline__ float to_f32(double x) {
  const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x);
  const int be = (int)((hi >> 20) & 0x7ff) - 896;
  const uint32_t m = (hi & 0x80000000u) | ((uint32_t)be << 23) | ((hi & 0xfffffu) << 3) | (lo >> 29);
  return be > 0 ? __uint_as_float(m) : 0.f;
}
__device__ __forceinline__ double to_f64(float f) {
  const uint32_t u = __float_as_uint(f), e = (u >> 23) & 0xff;
  return e ? __hiloint2double((int)((u & 0x80000000u) | ((((u >> 3) & 0x0fffffffu) + (896u << 20)))), (int)(u << 29)) : 0.0;
}
// v + part p of a b, b given as part_of_b(b, p)
__device__ __forceinline__ double2 part_of_b(double2 b, int p) { return p ? make_double2(b.y, b.x) : make_double2(b.x, -b.y); }
__device__ __forceinline__ double add_part(double2 a, double2 w, double v) { return fma(a.y, w.y, fma(a.x, w.x, v)); }
// part p of the complex product u z
__device__ __forceinline__ double mul_part(double2 u, double2 z, int p) {
  return fma(p ? u.y : -u.y, p ? z.x : z.y, u.x * (p ? z.y : z.x));
}

// 1 / d to FP64 accuracy, part p of it in lane parity p (a whole warp calls): an FP32 reciprocal y of d scaled
// into FP32's range (relative error r of about 2^-23), then y (1 + r + r^2) with r = 1 - d y in FP64 and
// r^2 in FP32 (the dropped r^3 is 2^-69).  An FP64 instruction of a warp takes 64 cycles of its SM
// partition whatever the lanes do: five of them here, a complex division is sixteen.  Pivots
// outside 2^(+-1000), zeros, Inf and NaN take the division.  (The off-diagonal tiles, like the sweeps and the FMA
// engine, divide by d through |d|^2, which needs |d| within 2^(+-511).)
__device__ __forceinline__ double recip_part(double dp, int p) {
  const double dq = shfl_d(dp, 1);
  const double dx = p ? dq : dp, dy = p ? dp : dq;
  const int m = max(exp_of(dx, 0), exp_of(dy, 0));
  if (__any_sync(0xffffffffu, m < 23 || m > 2023)) {
    const double2 v = cdiv(make_double2(1.0, 0.0), make_double2(dx, dy));
    return p ? v.y : v.x;
  }
  const int k = 1023 - m;                           // d 2^k: the larger part in [1, 2)
  const double ax = scale2(dx, k), ay = scale2(dy, k);
  const float fx = to_f32(ax), fy = to_f32(ay);
  const float n = 1.0f / (fx * fx + fy * fy);
  const float yx = fx * n, yy = -fy * n;
  const double dyx = to_f64(yx), dyy = to_f64(yy);
  double r = fma(-ax, p ? dyy : dyx, p ? 0.0 : 1.0);
  r = fma(p ? -ay : ay, p ? dyx : dyy, r);
  const double rq = shfl_d(r, 1);
  const double rx = p ? rq : r, ry = p ? r : rq;
  const float gx = to_f32(rx), gy = to_f32(ry);
  const float sx = gx * gx - gy * gy, sy = 2.f * gx * gy;          // r^2
  const float q = p ? yx * sy + yy * sx : yx * sx - yy * sy;       // y r^2
  double t = (p ? dyy : dyx) + to_f64(q);
  t = fma(dyx, p ? ry : rx, t);
  t = fma(p ? dyy : -dyy, p ? rx : ry, t);
  return scale2(t, k);
}

// Outputs of an update whose digit sum would fall short of FP64 (bit i: output (r0 + i, c)): ex, near, nz: scales, near
// and nonzero columns of the n products' rows [n][2 TB]
__device__ __noinline__ unsigned short_outputs(const short (*ex)[2 * TB], const unsigned long long* near, const unsigned long long* nz,
                                               int n, int r0, int c, const int* MA, const int* MB) {
  unsigned fix = 0;
#pragma unroll 1
  for (int i = 0; i < 16; ++i) {
    int best = E_NONE, rest = E_NONE;              // largest product of scales with a column near both, without
#pragma unroll 2
    for (int e = 0; e < n; ++e) {
      const int a = e * 2 * TB + r0 + i, b = e * 2 * TB + TB + c;
      const int ea = ex[e][r0 + i], eb = ex[e][TB + c];
      const bool hit = (near[a] & near[b]) != 0;
      if (hit && min(ea, eb) > E_ZERO) best = max(best, ea + eb);
      if (!hit && (nz[a] & nz[b])) rest = max(rest, ea + eb);       // rows that meet in zeros only: exactly zero
    }
    if (rest > best || (best > E_NONE && MA[r0 + i] + MB[c] - best > SPREAD)) fix |= 1u << i;
  }
  return fix;
}
// Outputs by FMAs.  solve: of S and X_JJ without its diagonal, else of the task's n products.
struct FixArgs {
  const TileTask* T;
  const KEntry* kl;
  const double2 *L, *Linv, *D, *E;                 // E: nullptr without pivoting
  const int* pm;
};
constexpr uint32_t FIX_B = TB * LDS * 16, FIX_LIST = 2 * FIX_B;  // operands [TB][LDS] (then the sums), list
constexpr int FIX_FEW = 64, FIX_MAX = 10 * NTHR;
static_assert(FIX_LIST + FIX_MAX * 2 <= SMEM_BYTES, "list of short outputs");
__device__ __forceinline__ double* fix_sum(unsigned char* smem) { return reinterpret_cast<double*>(smem); }
__device__ __forceinline__ unsigned short* fix_list(unsigned char* smem) { return reinterpret_cast<unsigned short*>(smem + FIX_LIST); }
// entries (row, k) of the operands of product e
__device__ __forceinline__ double2 fix_a(const FixArgs& g, const TileTask& T, bool solve, int e, int r, int k) {
  const int x = r * TB + k;
  if (!solve) return ld_cg(g.L + (int64_t)g.kl[T.kl_off + e].a_tile * TB * TB + x);
  const double* Sa = reinterpret_cast<const double*>(g.L + (int64_t)T.tile * TB * TB);
  return make_double2(__ldcg(Sa + x), __ldcg(Sa + TB * TB + x));
}
__device__ __forceinline__ double2 fix_b(const FixArgs& g, const TileTask& T, bool solve, int e, int r, int k) {
  const int x = r * TB + k;
  if (solve) return k == (g.E ? g.pm[r] : r) ? make_double2(0.0, 0.0) : ld_cg(g.Linv + (int64_t)T.col * TB * TB + x);
  const KEntry ke = g.kl[T.kl_off + e];
  const double2* b = g.L + (int64_t)ke.b_tile * TB * TB + x;
  double2 w = cmul(ld_cg(b), ld_cg(g.D + (int64_t)ke.kcol * TB + k));       // W_JK = L_JK D_K
  if (g.E) {
    const double2* eK = g.E + (int64_t)ke.kcol * TB + k;
    if (k + 1 < TB) w = cfma(ld_cg(b + 1), ld_cg(eK), w);
    if (k > 0) w = cfma(ld_cg(b - 1), ld_cg(eK - 1), w);
  }
  return w;
}
// the operands of product e in shared memory (all threads)
__device__ __noinline__ void stage_operands(const FixArgs& g, bool solve, int e, unsigned char* smem) {
  const TileTask T = *g.T;
  double2 *fA = reinterpret_cast<double2*>(smem), *fB = reinterpret_cast<double2*>(smem + FIX_B);
#pragma unroll 4
  for (int x = threadIdx.x; x < TB * TB; x += NTHR) {
    fA[(x >> 6) * LDS + (x & 63)] = fix_a(g, T, solve, e, x >> 6, x & 63);
    fB[(x >> 6) * LDS + (x & 63)] = fix_b(g, T, solve, e, x >> 6, x & 63);
  }
  __syncthreads();
}
// sums of the `count` <= FIX_MAX outputs of fix_list (part, row, column) into fix_sum (all threads)
__device__ __noinline__ void fma_outputs(const FixArgs& g, bool solve, int n, unsigned char* smem, int count) {
  if (count <= FIX_FEW) {                          // a warp an output (staging the tiles takes about 5 us a product)
    const TileTask T = *g.T;
    const int lane = threadIdx.x & 31;
#pragma unroll 1
    for (int q = threadIdx.x >> 5; q < count; q += NWK) {
      const int code = fix_list(smem)[q], r = code >> 6 & 63, c = code & 63;
      double v = 0.0;
#pragma unroll 2
      for (int e = 0; e < n; ++e)
#pragma unroll
        for (int k = lane; k < TB; k += 32) v = add_part(fix_a(g, T, solve, e, r, k), part_of_b(fix_b(g, T, solve, e, c, k), code >> 12), v);
      for (int o = 16; o > 0; o >>= 1) v += shfl_d(v, o);
      if (lane == 0) fix_sum(smem)[q] = v;
    }
    __syncthreads();
    return;
  }
  double v[FIX_MAX / NTHR];
#pragma unroll 1
  for (int e = 0; e < n; ++e) {
    stage_operands(g, solve, e, smem);
#pragma unroll 1
    for (int q = threadIdx.x, j = 0; q < count; q += NTHR, ++j) {
      const int code = fix_list(smem)[q];
      const double2* a = reinterpret_cast<const double2*>(smem) + (code >> 6 & 63) * LDS;
      const double2* b = reinterpret_cast<const double2*>(smem + FIX_B) + (code & 63) * LDS;
      double s = e ? v[j] : 0.0;
#pragma unroll 4
      for (int k = 0; k < TB; ++k) s = add_part(a[k], part_of_b(b[k], code >> 12), s);
      v[j] = s;
    }
    __syncthreads();
  }
  for (int q = threadIdx.x, j = 0; q < count; q += NTHR, ++j) fix_sum(smem)[q] = v[j];
  __syncthreads();
}

template <int V> struct IntC { static constexpr int value = V; };
using I4 = IntC<4>;
using I16 = IntC<16>;
using I64 = IntC<64>;

}  // namespace

// PIV: Bunch-Kaufman pivoting inside the diagonal tiles (diag_bk.cuh): Lt = P^T L, X = Lt^{-1} with its
// columns in the tile's own order, D with 2 x 2 blocks; the products are the same
template <bool PIV>
__global__ void __launch_bounds__(NTHR, 1) factor_dig_kernel(const FactorParams p) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* smem = smem_raw + ((1024u - (su(smem_raw) & 1023u)) & 1023u);
  __shared__ __align__(8) uint64_t bar_full[NSTG], bar_empty[NSTG], bar_accf, bar_acce;
  __shared__ uint32_t s_tmem;
  __shared__ int s_task, s_pending;
  __shared__ int s_MA[TB], s_MB[TB];              // largest row scales of the task's operands
  __shared__ const unsigned long long *s_fa[MAXP], *s_fb[MAXP];
  __shared__ const int4 *s_ea[MAXP], *s_eb[MAXP];
  __shared__ short s_ex[MAXP][2 * TB];            // row scales of every product of the task
  __shared__ int s_eL[TB], s_eW[TB];              // largest biased exponents of finished rows
  __shared__ unsigned s_near[TB][2], s_nearV[TB][2];   // columns near them (L or S, W)
  __shared__ unsigned s_nz[TB][2], s_nzV[TB][2];  // nonzero columns
  __shared__ unsigned s_nearL[TB], s_nearW[TB];   // the same of a panel product's operands: near, nonzero << 16
  __shared__ int s_pm[TB];                        // pivot mode: the tile's own order
  __shared__ int s_nfix, s_at;                    // short outputs of a task; listed so far
  __shared__ int s_ek[TB], s_eS[TB];              // balance of every column; the same in the tile's order
  __shared__ BkShared<double2> s_bk;              // pivot mode
  __shared__ double2 s_d[TB], s_dinv[TB], s_u[2][PW], s_x[2][PW], s_dg[2];
  __shared__ double2 sX[PW][PW + 1];              // inverse of a panel's diagonal block
  __shared__ float s_red[NWK];
  __shared__ int s_mexp[NWK];
  __shared__ double s_rec[TB];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (tid == 0) s_pending = -1;
  double2* Lg = reinterpret_cast<double2*>(p.L);
  double2* Linv = reinterpret_cast<double2*>(p.Linv);
  double2* Dg = reinterpret_cast<double2*>(p.D);
  unsigned long long* FL = reinterpret_cast<unsigned long long*>(p.opA);
  unsigned long long* FW = reinterpret_cast<unsigned long long*>(p.opB);
  int4* EL = p.rowA;
  int4* EW = p.rowB;
  uint2* ZL = p.nzA;
  uint2* ZW = p.nzB;
  constexpr int64_t TW = 2 * TB * TB;             // words of a tile

  if (tid == 0) {
    for (int s = 0; s < NSTG; ++s) {
      bar_init(su(&bar_full[s]), NWK);
      bar_init(su(&bar_empty[s]), 1);
    }
    bar_init(su(&bar_accf), 1);
    bar_init(su(&bar_acce), NWK);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(su(&s_tmem)), "r"(512u)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = s_tmem;
  uint32_t it = 0, tile_no = 0;                   // stages / products so far (same in every role)
  bool failed = false;

  // output of a worker thread: TMEM lane = embedded row (part ri, column c of the tile), 16 rows r0..
  const int tl = (warp & 3) * 32 + lane, ri = tl >> 6, oc = tl & 63, r0 = (warp >> 2) * 16;
  // operand item of a worker thread: threads 0..255 expand W, 256..511 L; row, part, half of a stage
  const int item = tid & 255, irow = item >> 2, ipart = (item >> 1) & 1, ik8 = item & 1;
  const bool iW = tid < 256;

  for (;;) {
    const int task = sched_pop(p, &s_task, &s_pending);
    if (task < 0) break;
    const TileTask T = p.tasks[task];
    const uint64_t deadline = globaltimer_ns() + (uint64_t)p.timeout_ns;
    const bool is_diag = (T.flags & TF_DIAG) != 0, is_upd = (T.flags & TF_UPDATE) != 0;
    const bool s_in = (T.flags & TF_S_IN) != 0;
    // the tile's accumulator (real parts, then imaginary parts) lies where L_IJ ends up: its last
    // reader, the final task, overwrites it
    double* Sa = reinterpret_cast<double*>(Lg + (int64_t)T.tile * TB * TB);
    double* sW = reinterpret_cast<double*>(smem);   // [2][64][LDS] results of a product (stages are idle then)

    long long H[16], Lo[16];
    // H, Lo += the levels (LS columns each) of the product in tensor memory, output i < NO from column
    // c0 + i of every level, shifted right by shift(i)
    auto read_levels = [&](auto no, auto ls, int c0, auto shift) {
#pragma unroll
      for (int jb = 0; jb < decltype(no)::value / 2; ++jb) {
        uint32_t v[NLV][2];
#pragma unroll
        for (int t = 0; t < NLV; ++t)
          tmem_ld2(tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)(t * decltype(ls)::value + c0 + jb * 2), v[t]);
        const int sh[2] = {shift(jb * 2), shift(jb * 2 + 1)};
        tmem_wait_ld(v);
#pragma unroll
        for (int q = 0; q < 2; ++q) {
          int l[NLV];
#pragma unroll
          for (int t = 0; t < NLV; ++t) l[t] = __float2int_rn(__uint_as_float(v[t][q]));
          // level t weighs 2^(-12 - 8 t) of the scales' product: u1 (levels 0..3, below 2^44)
          // in units of 2^-36, u2 (levels 4..7, below 2^49) in units of 2^-68
          const long long u1 = (long long)(l[0] * 256 + l[1]) * 65536 + (l[2] * 256 + l[3]);
          const long long u2 = (((long long)l[4] * 65536 + ((long long)l[5] * 256 + l[6])) << 8) + l[7];
          const int i = jb * 2 + q;
          const int s = min(sh[q], 62);
          if (__all_sync(0xffffffffu, s <= 10)) {      // nothing of u1 is shifted out
            H[i] += u1 << (10 - s);
            Lo[i] += (u2 << 6) >> s;
          } else {
            const long long a = u1 << 10;
            const long long hs = a >> s;
            const unsigned long long rem = (unsigned long long)a - ((unsigned long long)hs << s);
            H[i] += hs;
            Lo[i] += ((u2 << 6) >> s) + (long long)(s <= 28 ? rem << (28 - s) : rem >> (s - 28));
          }
        }
      }
    };
    // products of the n <= MAXP operand pairs listed in s_fa, s_fb (word pointers) and s_ea, s_eb (row
    // scales): H, Lo = sum of A B^T in units of 2^(MA[r] + MB[c] - 46), - 74; the outputs of the mask fix, whose
    // digits would fall short of FP64, by FMAs: in H as a double.  solve: the one pair is S and X_JJ without its
    // diagonal; the caller adds S (an output is short only if that term is small too).
    unsigned fix = 0;
    auto products = [&](int n, bool solve) {
      fix = 0;
#pragma unroll
      for (int i = 0; i < 16; ++i) H[i] = Lo[i] = 0;
      Words8 w;
      auto fetch_words = [&](int c) {
        w = load_words((iW ? s_fb : s_fa)[c / NCH] + ((c % NCH) * 256 + item) * 8);
      };
      fetch_words(0);
      unsigned long long* near = reinterpret_cast<unsigned long long*>(smem);   // [n][2 TB] (the stages are idle)
      bool look = false;
      if (tid == 0) s_nfix = s_at = 0;
      const uint2 zx = solve ? __ldcg(ZL + (s_eb[0] - EL) + oc) : make_uint2(0, 0);   // nonzero columns of row oc of X_JJ
#pragma unroll 2
      for (int i = tid; i < n * 2 * TB; i += NTHR) {
        const int e = i >> 7, q = i & 127;
        const int4 row = __ldcg((q < TB ? s_ea[e] : s_eb[e]) + (q & 63));
        s_ex[e][q] = (short)row.x;
        near[i] = (unsigned)row.z | (unsigned long long)(unsigned)row.w << 32;
      }
      __syncthreads();
      // every two rows share a near column (rows of zeros have all bits; both parts' threads hold the same
      // outputs, so each looks at half of them)
      if (!solve) {
#pragma unroll 1
        for (int e = 0; e < n; ++e) {
          const uint2 b = *reinterpret_cast<const uint2*>(near + e * 2 * TB + TB + oc);
          const uint4* a = reinterpret_cast<const uint4*>(near + e * 2 * TB + r0 + 8 * ri);
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const uint4 v = a[i];
            look |= ((v.x & b.x) | (v.y & b.y)) == 0 || ((v.z & b.x) | (v.w & b.y)) == 0;
          }
        }
      }
      // the largest scale of every operand row over the task
      if (tid < 2 * TB) {
        int m = E_ZERO, lo = E_BAD;
        for (int e = 0; e < n; ++e) {
          m = max(m, (int)s_ex[e][tid]);
          lo = min(lo, (int)s_ex[e][tid]);
        }
        (tid < TB ? s_MA : s_MB)[tid & 63] = m;
        look |= m > E_ZERO && lo < m - SPREAD / 2;
      }
      const bool looked = __syncthreads_or(look || solve);
      int nst = n * NCH;
      if (looked) {
        if (solve) {
          const short2* old = reinterpret_cast<const short2*>(smem + OLD_OFF) + (PIV ? s_pm[oc] : oc);
          const unsigned long long nb = near[TB + oc];
          const int eb = s_MB[oc];
#pragma unroll 2
          for (int i = 0; i < 16; ++i) {
            const short2 o = old[(r0 + i) * TB];
            const bool meet = (s_nz[r0 + i][0] & zx.x) | (s_nz[r0 + i][1] & zx.y);
            if (!(near[r0 + i] & nb) && meet && max(o.x, o.y) - 1022 + SLACK < s_MA[r0 + i] + eb) fix |= 1u << i;
          }
        } else {
          unsigned long long* nz = reinterpret_cast<unsigned long long*>(smem + OLD_OFF);   // [n][2 TB]
          for (int i = tid; i < n * 2 * TB; i += NTHR) {
            const int e = i >> 7, q = i & 127;
            const uint2 z = __ldcg(q < TB ? ZL + (s_ea[e] - EL) + q : ZW + (s_eb[e] - EW) + q - TB);
            nz[i] = z.x | (unsigned long long)z.y << 32;
          }
          __syncthreads();
          fix = short_outputs(s_ex, near, nz, n, r0, oc, s_MA, s_MB);
        }
        if (fix) atomicAdd(&s_nfix, __popc(fix));
        __syncthreads();
        // most of them (over FIX_MAX of 8192): all by FMAs, which takes 0.6 of the list's time an output (groups above:
        // half of the outputs 250 ms by the list, 312 all)
        if (s_nfix > FIX_MAX) nst = 0;
      }
      const uint32_t it0 = it, tile0 = tile_no;
      // one thread: the MMAs of stage c
      auto issue = [&](int c) {
        const uint32_t s = (it0 + c) % NSTG, use = (it0 + c) / NSTG;
        const uint32_t tn = tile0 + c / NCH;
        if (c % NCH == 0 && !bar_wait(su(&bar_acce), (tn & 1) ^ 1, deadline)) { failed = true; return; }
        if (!bar_wait(su(&bar_full[s]), use & 1, deadline)) { failed = true; return; }
        fence_after();
        stage_mmas<TB>(tmem, su(smem + s * STAGE), c % NCH == 0);
        mma_commit(su(&bar_empty[s]));
        if (c % NCH == NCH - 1) mma_commit(su(&bar_accf));
      };
      // the first stage of a product is expanded before the read-back of the product before it, which
      // frees the tensor memory for its MMAs; the second one while those run
      for (int c = 0; c <= nst && !failed; ++c) {
        if (c < nst) {
          const uint32_t s = (it0 + c) % NSTG, use = (it0 + c) / NSTG;
          failed = !__all_sync(0xffffffffu, bar_wait(su(&bar_empty[s]), (use & 1) ^ 1, deadline));
          if (failed) break;
          put_digits(smem + s * STAGE, iW, irow, ipart, ik8, w);
          if (c + 1 < nst) fetch_words(c + 1);
          asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
          __syncwarp();
          if (lane == 0) bar_arrive(su(&bar_full[s]));
          if (warp == ISSUER && (c < NCH || c % NCH != 0)) {
            if (lane == 0) issue(c);
            failed = __any_sync(0xffffffffu, failed);
          }
        }
        if (c >= NCH && c % NCH == 0) {
          // ---- read back the levels of product e
          const int e = c / NCH - 1;
          const int db = s_MB[oc] - s_ex[e][TB + oc];
          failed = !__all_sync(0xffffffffu, bar_wait(su(&bar_accf), tile_no & 1, deadline));
          if (failed) break;
          fence_after();
          read_levels(I16{}, I64{}, r0, [&](int i) { return s_MA[r0 + i] - s_ex[e][r0 + i] + db; });
          fence_before();
          __syncwarp();
          if (lane == 0) bar_arrive(su(&bar_acce));
          ++tile_no;
          if (warp == ISSUER && (e + 1) * NCH < nst) {
            if (lane == 0) issue((e + 1) * NCH);
            failed = __any_sync(0xffffffffu, failed);
          }
        }
      }
      it = it0 + nst;
      if (looked && s_nfix) {
        const FixArgs g{p.tasks + task, p.klist, Lg, Linv, Dg, PIV ? reinterpret_cast<const double2*>(p.E) : nullptr, s_pm};
        __syncthreads();                           // the last levels are read: the stages are free
        if (nst == 0) {
          fix = 0xffff;
          const double2 *a = reinterpret_cast<const double2*>(smem) + r0 * LDS, *b = reinterpret_cast<const double2*>(smem + FIX_B) + oc * LDS;
#pragma unroll 1
          for (int e = 0; e < n; ++e) {
            stage_operands(g, solve, e, smem);
#pragma unroll
            for (int i = 0; i < 16; i += 4) {
              double v[4];
#pragma unroll
              for (int u = 0; u < 4; ++u) v[u] = __longlong_as_double(H[i + u]);
#pragma unroll 2
              for (int k = 0; k < TB; ++k) {
                const double2 w = part_of_b(b[k], ri);
#pragma unroll
                for (int u = 0; u < 4; ++u) v[u] = add_part(a[(i + u) * LDS + k], w, v[u]);
              }
#pragma unroll
              for (int u = 0; u < 4; ++u) H[i + u] = __double_as_longlong(v[u]);
            }
            __syncthreads();
          }
        } else {
          const int q0 = fix ? atomicAdd(&s_at, __popc(fix)) : 0;
          int q = q0;
#pragma unroll 1
          for (unsigned f = fix; f; f &= f - 1) fix_list(smem)[q++] = (unsigned short)(ri << 12 | (r0 + __ffs(f) - 1) << 6 | oc);
          __syncthreads();
          fma_outputs(g, solve, n, smem, s_nfix);
          q = q0;
#pragma unroll
          for (int i = 0; i < 16; ++i)
            if (fix >> i & 1) H[i] = __double_as_longlong(fix_sum(smem)[q++]);
          __syncthreads();
        }
      }
    };
    auto result = [&](int i) -> double {
      return fix >> i & 1 ? __longlong_as_double(H[i]) : fixed_to_double<28>(H[i], Lo[i], s_MA[r0 + i] + s_MB[oc] - 74);
    };

    // ---------------------------------------------------------------- 1. Schur products
    if (T.nk > 0) {
      if (tid < T.nk) {
        const KEntry ke = p.klist[T.kl_off + tid];
        s_fa[tid] = FL + (int64_t)ke.a_tile * TW;
        s_fb[tid] = FW + (int64_t)ke.b_tile * TW;
        s_ea[tid] = EL + (int64_t)ke.a_tile * TB;
        s_eb[tid] = EW + (int64_t)ke.b_tile * TB;
      }
      __syncthreads();
      products(T.nk, false);
    }
    if (__syncthreads_or(failed)) {
      if (tid == 0) set_error(p.ctl, D3M_ERR_TIMEOUT, task);
      break;
    }
    trace_mark(p, task, 0);
    // S = S_in - products (this thread: part ri of column oc, rows r0 ..)
    double S[16];
    {
#pragma unroll
      for (int i = 0; i < 16; ++i) {
        if (s_in) {
          S[i] = __ldcg(Sa + ri * TB * TB + (r0 + i) * TB + oc);
        } else {
          const double2 k = k_entry<double>(T, p.K, r0 + i, oc);
          S[i] = ri ? k.y : k.x;
        }
      }
      if (T.nk > 0) {
#pragma unroll
        for (int i = 0; i < 16; ++i) S[i] -= result(i);
      }
    }
    if (is_upd) {
      {
#pragma unroll
        for (int i = 0; i < 16; ++i) Sa[ri * TB * TB + (r0 + i) * TB + oc] = S[i];
      }
      sched_complete(p, task);
      continue;
    }
    __syncthreads();                                // s_MA, s_MB and the stages are free
    if (is_diag) {
      // -------------------------------------------------------------- 2a. diagonal tile
      // Unpivoted LDL^T and X = L^{-1} in panels of 16 columns, S and L in the lower triangle of sS, X
      // transposed in the upper one (sS[s][r] = X[r][s], first its sum Z).  Panel k: the 16 x 16
      // diagonal block in FP64 (a chain of 16 pivots); V = sS[:, panel] X_kk^T for all other rows
      // (below: W, above: -X); then T[r][s] -= L[r][:] U[s][:] for the rows r below and s <= r,
      // U = V outside the panel and -X_kk inside.  Both are digit products of one stage: the FP64
      // pipe would take three times as long for them.
      double2* sS = reinterpret_cast<double2*>(smem + SMEM_S);
      double* sV = reinterpret_cast<double*>(smem + SMEM_S + TB * LDS * 16);   // [2][64][PW + 1]
#pragma unroll
      for (int i = 0; i < 16; ++i) {
        const int r = r0 + i;
        reinterpret_cast<double*>(sS + r * LDS + oc)[ri] = oc <= r ? S[i] : 0.0;
      }
      __syncthreads();
      const int nr = T.rv;                          // real unknowns of the tile
      // max |S| over the real lower triangle (breakdown scale), in FP32 relative to the largest exponent; Inf if an
      // entry is, and a NaN does not count
      auto mag_exp = [](double2 z) {
        const int e = max(exp_of(z.x, 0), exp_of(z.y, 0));
        return e >= X_BAD && (isnan(z.x) || isnan(z.y)) ? X_ZERO : e;
      };
      int mexp = X_ZERO;
      for (int i = tid; i < TB * TB; i += NTHR) {
        const int r = i >> 6, c = i & 63;
        if (c <= r && r < nr) mexp = max(mexp, mag_exp(sS[r * LDS + c]));
      }
      mexp = __reduce_max_sync(0xffffffffu, mexp);
      if (lane == 0) s_mexp[warp] = mexp;
      __syncthreads();
#pragma unroll
      for (int w = 0; w < NWK; ++w) mexp = max(mexp, s_mexp[w]);
      {
        float mx = 0.f;
        for (int i = tid; i < TB * TB; i += NTHR) {
          const int r = i >> 6, c = i & 63;
          if (c <= r && r < nr && mag_exp(sS[r * LDS + c]) != X_ZERO) {
            const float x = to_f32(scale2(sS[r * LDS + c].x, 1023 - mexp)), y = to_f32(scale2(sS[r * LDS + c].y, 1023 - mexp));
            mx = fmaxf(mx, x * x + y * y);
          }
        }
        for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        if (lane == 0) s_red[warp] = mx;
      }
      if constexpr (PIV) {
        bk_factor<double, NTHR>(sS, LDS, s_bk);
      } else {
      // one digit product of operands in shared memory (16 columns, nrow rows of the L side):
      // value(w_side, row, q, part) 2^(-+ balance of column q) (W side -, L side +)
      auto local_product = [&](auto nrow, int c0, auto value) {
        constexpr int NR = decltype(nrow)::value;
        if (iW || irow < NR) {
          double v[8];
          int m = X_ZERO, sh[8], ex[8];
#pragma unroll
          for (int e = 0; e < 8; ++e) {
            const int q = ik8 * 8 + e;
            v[e] = value(iW, irow, q, ipart);
            sh[e] = iW ? -s_ek[c0 + q] : s_ek[c0 + q];
            ex[e] = exp_of(v[e], sh[e]);
            m = max(m, ex[e]);
          }
          m = max(m, __shfl_xor_sync(0xffffffffu, m, 1));
          m = max(m, __shfl_xor_sync(0xffffffffu, m, 2));
          const int E = row_scale(m);
          unsigned nb = 0;                        // the row's columns near its largest entry
#pragma unroll
          for (int e = 0; e < 8; ++e) nb |= ((unsigned)near_max(ex[e], m) | (unsigned)(ex[e] != X_ZERO) << 16) << e;
          nb <<= ik8 * 8;
          nb |= __shfl_xor_sync(0xffffffffu, nb, 1);
          nb |= __shfl_xor_sync(0xffffffffu, nb, 2);
          if ((item & 3) == 0) {
            (iW ? s_MB : s_MA)[irow] = E;
            (iW ? s_nearW : s_nearL)[irow] = no_near(E) ? (nb & 0xffff0000u) | (E >= E_BAD ? 0xffff0000u : 0) : (m <= X_ZERO ? ~0u : nb);
          }
          Words8 w;
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            w.w[e].x = word_of(v[2 * e], sh[2 * e], E);
            w.w[e].y = word_of(v[2 * e + 1], sh[2 * e + 1], E);
          }
          put_digits<NR>(smem, iW, irow, ipart, ik8, w);
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncthreads();
        if (tid == 0) {
          if (!bar_wait(su(&bar_acce), (tile_no & 1) ^ 1, deadline)) failed = true;
          else {
            fence_after();
            stage_mmas<NR>(tmem, su(smem), true);
            mma_commit(su(&bar_accf));
          }
        }
        __syncwarp();
        if (!bar_wait(su(&bar_accf), tile_no & 1, deadline)) failed = true;
        failed = __syncthreads_or(failed);
        fence_after();
#pragma unroll
        for (int i = 0; i < 16; ++i) H[i] = Lo[i] = 0;
      };
      // output (r, oc) of a local product, a term of a sum that starts at `old`: whether it needs FMAs, and their sum
      auto local_short = [&](int r, double old) -> bool {
        const unsigned both = s_nearL[r] & s_nearW[oc];     // rows that meet in zeros only: exactly zero
        return both >= 0x10000u && !(both & 0xffffu) && exp_of(old, 0) - 1022 + SLACK < s_MA[r] + s_MB[oc];
      };
      auto local_fma = [&](int r, auto value) -> double {
        double s = 0.0;
#pragma unroll 1
        for (int q = 0; q < PW; ++q)
          s = add_part(make_double2(value(false, r, q, 0), value(false, r, q, 1)), part_of_b(make_double2(value(true, oc, q, 0), value(true, oc, q, 1)), ri), s);
        return s;
      };
      auto product_read = [&]() {
        fence_before();
        __syncwarp();
        if (lane == 0) bar_arrive(su(&bar_acce));
        ++tile_no;
      };
      // part ep of element (er, es), es <= er, of a panel's diagonal block: one per thread of nine warps
      // of SM partitions 1..3; warp 0 (partition 0) runs the chain of pivots
      const int ew = (warp & 3) ? (warp >> 2) * 3 + (warp & 3) - 1 : 99;
      const int eidx = (ew * 32 + lane) >> 1, ep = lane & 1;
      const bool lwarp = warp == 0 || ew < 9;
      int er = 0;
      while (er < PW && (er + 1) * (er + 2) / 2 <= eidx) ++er;
      const int es = eidx - er * (er + 1) / 2;
      const bool live = er < PW;
      for (int c0 = 0; c0 < nr && !failed; c0 += PW) {
        if (lwarp) {
          auto part_of = [](double2* z, int q) -> double& { return reinterpret_cast<double*>(z)[q]; };
          double v = (live && warp) ? part_of(sS + (c0 + er) * LDS + c0 + es, ep) : 0.0;
          // state before step c: u = column c of S (rows >= c), x = row c of X, the pivot and its
          // reciprocal, and the next diagonal entry before the update of step c
          if (warp == 0) {
            const double d0 = part_of(sS + c0 * LDS + c0, ep);
            const double di = recip_part(d0, ep);
            if (lane < 2) {
              part_of(s_d + c0, ep) = d0;
              part_of(s_dinv + c0, ep) = di;
            }
          } else if (live) {
            if (es == 0) part_of(&s_u[0][er], ep) = v;
            if (er == 1 && es == 1) part_of(&s_dg[0], ep) = v;
          }
          asm volatile("bar.sync 1, 320;" ::: "memory");
          for (int c = 0; c < PW; ++c) {
            const int pb = c & 1;
            const double2 di = s_dinv[c0 + c];
            if (warp == 0) {
              if (c + 1 < PW) {
                const double2 u = s_u[pb][c + 1], dg = s_dg[pb];
                // l = u / d, d_(c+1) = dg - l u, its reciprocal
                const double lp = mul_part(u, di, ep);
                const double lq = shfl_d(lp, 1);
                const double lx = ep ? lq : lp, ly = ep ? lp : lq;
                double d = fma(-lx, ep ? u.y : u.x, ep ? dg.y : dg.x);
                d = fma(ep ? -ly : ly, ep ? u.x : u.y, d);
                const double rp = recip_part(d, ep);
                if (lane < 2) {
                  part_of(s_d + c0 + c + 1, ep) = d;
                  part_of(s_dinv + c0 + c + 1, ep) = rp;
                }
              }
            } else if (__any_sync(0xffffffffu, live && er > c)) {
              const double2 u = s_u[pb][live && er > c ? er : PW - 1];
              const double lp = mul_part(u, di, ep);
              const double lq = shfl_d(lp, 1);
              const double lx = ep ? lq : lp, ly = ep ? lp : lq;
              // S[r][s] -= l S[s][c] (s > c), X[r][s] -= l X[c][s] (s < c), X[r][c] = -l
              const double2 t = es > c ? s_u[pb][live ? es : 0] : s_x[pb][live ? es : 0];
              double n = fma(-lx, ep ? t.y : t.x, v);
              n = fma(ep ? -ly : ly, ep ? t.x : t.y, n);
              if (live && er > c) {
                if (es == c) part_of(sS + (c0 + er) * LDS + c0 + c, ep) = lp;
                v = es == c ? -lp : n;
              }
            }
            if (warp && live) {
              if (es == c + 1) part_of(&s_u[pb ^ 1][er], ep) = v;
              if (er == c + 1 && es <= c) part_of(&s_x[pb ^ 1][es], ep) = v;
              if (er == c + 2 && es == c + 2) part_of(&s_dg[pb ^ 1], ep) = v;
            }
            asm volatile("bar.sync 1, 320;" ::: "memory");
          }
          if (warp && live) {
            part_of(&sX[er][es], ep) = er == es ? (ep ? 0.0 : 1.0) : v;
            if (er != es) {
              part_of(&sX[es][er], ep) = 0.0;
              part_of(sS + (c0 + es) * LDS + c0 + er, ep) = v;
            }
          }
          if (warp == 0 && lane < PW) s_ek[c0 + lane] = balance_of(s_d[c0 + lane]);
        }
        __syncthreads();
        const int c1 = c0 + PW;
        // V = sS[:, panel] X_kk^T, rows outside the panel: the W side holds the 64 rows, the L side
        // X_kk without its diagonal, so a thread reads back 4 columns of row oc
        auto v_value = [&](bool ws, int row, int q, int part) -> double {
          if (!ws) return row != q ? reinterpret_cast<const double*>(&sX[row][q])[part] : 0.0;
          return (row < c0 || row >= c1) ? reinterpret_cast<const double*>(sS + row * LDS + c0 + q)[part] : 0.0;
        };
        local_product(I16{}, c0, v_value);
        if (failed) break;
        {
          const int q0 = (warp >> 2) * 4;
          read_levels(I4{}, I16{}, q0, [](int) { return 0; });
          product_read();
          const double* old = reinterpret_cast<const double*>(sS + oc * LDS + c0 + q0) + ri;
          double* v = sV + (ri * TB + oc) * (PW + 1) + q0;
          unsigned fl = 0;
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            v[i] = old[2 * i] + fixed_to_double<28>(H[i], Lo[i], s_MA[q0 + i] + s_MB[oc] - 74);
            if (local_short(q0 + i, old[2 * i])) fl |= 1u << i;
          }
#pragma unroll 1
          for (; fl; fl &= fl - 1) {
            const int i = __ffs(fl) - 1;
            v[i] = old[2 * i] + local_fma(q0 + i, v_value);
          }
        }
        __syncthreads();
        // above the panel X = -V, below L = V / d
        for (int i = tid; i < TB * PW; i += NTHR) {
          const int r = i >> 4, q = i & (PW - 1);
          const double2 v = make_double2(sV[r * (PW + 1) + q], sV[(TB + r) * (PW + 1) + q]);
          if (r < c0) sS[r * LDS + c0 + q] = make_double2(-v.x, -v.y);
          else if (r >= c1) sS[r * LDS + c0 + q] = cmul(v, s_dinv[c0 + q]);
        }
        __syncthreads();
        if (c1 >= nr) break;
        // (U inside the panel without the diagonal of -X_kk: L[r][s] itself is added to Z[r][s], which is zero there)
        auto t_value = [&](bool ws, int row, int q, int part) -> double {
          if (!ws) return row >= c1 ? reinterpret_cast<const double*>(sS + row * LDS + c0 + q)[part] : 0.0;
          if (row < c0 || row >= c1) return sV[(part * TB + row) * (PW + 1) + q];
          return q != row - c0 ? -reinterpret_cast<const double*>(&sX[q][row - c0])[part] : 0.0;
        };
        local_product(I64{}, c0, t_value);
        if (failed) break;
        // rows c1 .. 63 in groups of 4, a quarter of them to each of the four warps of an SM partition
        {
          const int per = (TB - c1) >> 2, rw = c1 + (warp >> 2) * per;
#pragma unroll 1
          for (int rb = rw; rb < rw + per; rb += 4) {
#pragma unroll
            for (int i = 0; i < 4; ++i) H[i] = Lo[i] = 0;
            read_levels(I4{}, I64{}, rb, [](int) { return 0; });
            unsigned fl = 0;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              const int r = rb + i;
              if (oc <= r) {
                double* t = reinterpret_cast<double*>(oc >= c1 ? sS + r * LDS + oc : sS + oc * LDS + r) + ri;
                const double old = oc >= c0 && oc < c1 ? reinterpret_cast<const double*>(sS + r * LDS + oc)[ri] : *t;
                if (!local_short(r, old)) *t = old - fixed_to_double<28>(H[i], Lo[i], s_MA[r] + s_MB[oc] - 74);
                else fl |= 1u << i;
              }
            }
#pragma unroll 1
            for (; fl; fl &= fl - 1) {
              const int r = rb + __ffs(fl) - 1;
              double* t = reinterpret_cast<double*>(oc >= c1 ? sS + r * LDS + oc : sS + oc * LDS + r) + ri;
              const double old = oc >= c0 && oc < c1 ? reinterpret_cast<const double*>(sS + r * LDS + oc)[ri] : *t;
              *t = old - local_fma(r, t_value);
            }
          }
        }
        product_read();
        __syncthreads();
      }
      }
      if (__syncthreads_or(failed)) {
        if (tid == 0) set_error(p.ctl, D3M_ERR_TIMEOUT, task);
        break;
      }
      if constexpr (PIV) {
        if (tid < TB) {
          s_d[tid] = s_bk.d[tid];
          // a 2 x 2 block's two columns share the balance of its largest entry
          double2 m = s_bk.d[tid];
          const bool first2 = s_bk.e[tid].x != 0 || s_bk.e[tid].y != 0;
          const bool second2 = tid > 0 && (s_bk.e[tid - 1].x != 0 || s_bk.e[tid - 1].y != 0);
          s_ek[tid] = pair_balance(m, first2 ? s_bk.d[tid + 1] : (second2 ? s_bk.d[tid - 1] : m),
                                   first2 ? s_bk.e[tid] : (second2 ? s_bk.e[tid - 1] : m));
        }
      } else if (tid < TB && tid >= nr) {
        // rows of padding are rows of the identity
        s_d[tid] = make_double2(1.0, 0.0);
        s_ek[tid] = 0;
      }
      __syncthreads();
      trace_mark(p, task, 2);
      {
        double2* Li = Linv + (int64_t)T.col * TB * TB;
        unsigned long long* f = FL + (int64_t)T.tile * TW;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int r = warp + 16 * i;
          double2 x[2];
          int m = X_ZERO, ex[2];
#pragma unroll
          for (int q = 0; q < 2; ++q) {
            const int s = lane + 32 * q;
            x[q] = (s < r && (PIV || r < nr)) ? sS[s * LDS + r] : make_double2(0.0, 0.0);
            ex[q] = max(exp_of(x[q].x, s_ek[s]), exp_of(x[q].y, s_ek[s]));
            m = max(m, ex[q]);
          }
          m = __reduce_max_sync(0xffffffffu, m);
          const int E = row_scale(m);
          unsigned near0 = 0, near1 = 0, nz0 = 0, nz1 = 0;
#pragma unroll
          for (int q = 0; q < 2; ++q) {
            const int s = lane + 32 * q, k = PIV ? s_bk.perm[s] : s;   // column k of X = Lt^{-1}; words without its diagonal
            Li[r * TB + k] = s == r ? make_double2(1.0, 0.0) : x[q];
            f[word_at(r, k, 0)] = word_of(x[q].x, s_ek[s], E);
            f[word_at(r, k, 1)] = word_of(x[q].y, s_ek[s], E);
            if (near_max(ex[q], m)) (k < 32 ? near0 : near1) |= 1u << (k & 31);
            if (ex[q] != X_ZERO) (k < 32 ? nz0 : nz1) |= 1u << (k & 31);
          }
          near0 = __reduce_or_sync(0xffffffffu, near0);
          near1 = __reduce_or_sync(0xffffffffu, near1);
          nz0 = __reduce_or_sync(0xffffffffu, nz0);
          nz1 = __reduce_or_sync(0xffffffffu, nz1);
          if (lane == 0) {
            EL[(int64_t)T.tile * TB + r] = row_info(m, near0, near1);
            ZL[(int64_t)T.tile * TB + r] = row_nonzero(m, nz0, nz1);
          }
        }
        double2* Lt = Lg + (int64_t)T.tile * TB * TB;
        for (int i = tid; i < TB * TB; i += NTHR) {
          const int r = i >> 6, c = i & 63;
          Lt[(PIV ? s_bk.perm[r] : r) * TB + c] = (c < r && (PIV || r < nr)) ? sS[r * LDS + c] : make_double2(c == r ? 1.0 : 0.0, 0.0);
        }
        if (tid < TB) {
          Dg[(int64_t)T.col * TB + tid] = s_d[tid];
          if (PIV) {
            reinterpret_cast<double2*>(p.E)[(int64_t)T.col * TB + tid] = s_bk.e[tid];
            p.piv[(int64_t)T.col * TB + tid] = s_bk.perm[tid];
          }
        }
        if (warp == 0) {
          float smx = 0.f;
          for (int w = 0; w < NWK; ++w) smx = fmaxf(smx, s_red[w]);
          const double smax = mexp >= X_BAD ? (double)INFINITY : scale2((double)sqrtf(smx), mexp - 1023);
          double amin = 3.0e38, amax = 0.0;
          if constexpr (PIV) {
            bk_pivot_range<double>(s_bk, T.cv, amin, amax);
          } else {
            for (int c = lane; c < T.cv; c += 32) {
              const double a = sqrt(cabs2(s_d[c]));
              amin = fmin(amin, a);
              amax = fmax(amax, a);
            }
            for (int o = 16; o > 0; o >>= 1) {
              amin = fmin(amin, __shfl_xor_sync(0xffffffffu, amin, o));
              amax = fmax(amax, __shfl_xor_sync(0xffffffffu, amax, o));
            }
          }
          if (lane == 0) {
            record_pivot_stats(p.ctl, (float)amin, (float)amax);
            if (!(amin >= p.piv_tol * smax)) set_error(p.ctl, D3M_ERR_PIVOT, task);
          }
        }
      }
    } else {
      // -------------------------------------------------------------- 2b. off-diagonal tile
      // W_IJ = S X^T = S + S (X - I)^T with the words of S in this tile's own slot, then L_IJ = W_IJ / d
      unsigned long long* f = FL + (int64_t)T.tile * TW;
      if (tid < TB) {
        s_eL[tid] = X_ZERO;
        s_eW[tid] = X_ZERO;
        s_near[tid][0] = s_near[tid][1] = s_nz[tid][0] = s_nz[tid][1] = 0;
        const double2 d = ld_cg(Dg + (int64_t)T.col * TB + tid);
        s_d[tid] = d;
        if constexpr (PIV) {
          // D^{-1}: [w_c w_(c+1)] [[d1, e], [e, d2]]^{-1}; s_u2 = the weight of the other column of a block
          const double2* Eg = reinterpret_cast<const double2*>(p.E) + (int64_t)T.col * TB;
          const double2 zero = make_double2(0.0, 0.0);
          const double2 e0 = ld_cg(Eg + tid), e1 = tid > 0 ? ld_cg(Eg + tid - 1) : zero;
          const bool first2 = e0.x != 0 || e0.y != 0, second2 = e1.x != 0 || e1.y != 0;
          const double2 o = first2 || second2 ? ld_cg(Dg + (int64_t)T.col * TB + (first2 ? tid + 1 : tid - 1)) : d;
          const double2 e = first2 ? e0 : (second2 ? e1 : zero);
          const double2 det = first2 || second2 ? csub(cmul(d, o), cmul(e, e)) : d;
          s_bk.u1[tid] = first2 || second2 ? cdiv(o, det) : cdiv(make_double2(1.0, 0.0), d);
          s_bk.u2[tid] = first2 || second2 ? cdiv(make_double2(-e.x, -e.y), det) : zero;
          s_bk.perm[tid] = first2 ? tid + 1 : (second2 ? tid - 1 : tid);
          const int bal = pair_balance(d, o, first2 || second2 ? e : d);
          s_ek[tid] = bal;
          // the contraction of the triangular solve runs over the tile's own order
          s_pm[tid] = p.piv[(int64_t)T.col * TB + tid];
          s_eS[s_pm[tid]] = bal;
        } else {
          s_ek[tid] = s_eS[tid] = balance_of(d);
          s_rec[tid] = 1.0 / (d.x * d.x + d.y * d.y);
        }
      }
      __syncthreads();
      {
        const int bal = s_eS[oc];
#pragma unroll
        for (int i = 0; i < 16; ++i) {
          const int m = __reduce_max_sync(0xffffffffu, exp_of(S[i], -bal));
          if (lane == 0) atomicMax(&s_eL[r0 + i], m);
        }
        __syncthreads();
#pragma unroll
        for (int i = 0; i < 16; ++i) {
          const int m = s_eL[r0 + i];
          f[word_at(r0 + i, oc, ri)] = word_of(S[i], -bal, row_scale(m));
          if (!s_in) Sa[ri * TB * TB + (r0 + i) * TB + oc] = S[i];   // read again after the product
          reinterpret_cast<short*>(smem + OLD_OFF)[((r0 + i) * TB + oc) * 2 + ri] = (short)exp_of(S[i], 0);
          const unsigned near = __ballot_sync(0xffffffffu, near_max(exp_of(S[i], -bal), m));
          const unsigned nz = __ballot_sync(0xffffffffu, m <= X_ZERO || m >= X_BAD || exp_of(S[i], 0) != X_ZERO);
          if (lane == 0) {
            atomicOr(&s_near[r0 + i][warp & 1], near);
            atomicOr(&s_nz[r0 + i][warp & 1], nz);
          }
        }
      }
      __syncthreads();
      if (tid < TB) {
        EL[(int64_t)T.tile * TB + tid] = row_info(s_eL[tid], s_near[tid][0], s_near[tid][1]);
        s_eL[tid] = X_ZERO;
      }
      if (tid == 0) {
        s_fa[0] = f;
        s_fb[0] = FL + (int64_t)T.diag * TW;
        s_ea[0] = EL + (int64_t)T.tile * TB;
        s_eb[0] = EL + (int64_t)T.diag * TB;
      }
      __syncthreads();
      trace_mark(p, task, 1);
      products(1, true);
      if (__syncthreads_or(failed)) {
        if (tid == 0) set_error(p.ctl, D3M_ERR_TIMEOUT, task);
        break;
      }
      {
#pragma unroll
        for (int i = 0; i < 16; ++i) sW[(ri * TB + r0 + i) * LDS + oc] = __ldcg(Sa + ri * TB * TB + (r0 + i) * TB + (PIV ? s_pm[oc] : oc)) + result(i);
      }
      __syncthreads();
      trace_mark(p, task, 2);
      // thread: column c, rows wr + 8 i (a warp holds half a row)
      const int c = tid & 63, wr = tid >> 6, bal = s_ek[c];
      double2 w[8], l[8];
      {
        const double2 d = s_d[c];
        const double rec = s_rec[c];
        double2* Lt = Lg + (int64_t)T.tile * TB * TB;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const int r = wr + 8 * i;
          w[i] = make_double2(sW[r * LDS + c], sW[(TB + r) * LDS + c]);
          if constexpr (PIV) {
            const int o = s_bk.perm[c];
            l[i] = cfma(make_double2(sW[r * LDS + o], sW[(TB + r) * LDS + o]), s_bk.u2[c], cmul(w[i], s_bk.u1[c]));
          } else {
            l[i] = make_double2((w[i].x * d.x + w[i].y * d.y) * rec, (w[i].y * d.x - w[i].x * d.y) * rec);
          }
          Lt[r * TB + c] = l[i];
          const int bw = __reduce_max_sync(0xffffffffu, max(exp_of(w[i].x, -bal), exp_of(w[i].y, -bal)));
          const int bl = __reduce_max_sync(0xffffffffu, max(exp_of(l[i].x, bal), exp_of(l[i].y, bal)));
          if (lane == 0) {
            atomicMax(&s_eW[r], bw);
            atomicMax(&s_eL[r], bl);
          }
        }
      }
      __syncthreads();
      {
        unsigned long long* g = FW + (int64_t)T.tile * TW;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const int r = wr + 8 * i;
          const int eW = row_scale(s_eW[r]), eL = row_scale(s_eL[r]);
          f[word_at(r, c, 0)] = word_of(l[i].x, bal, eL);
          f[word_at(r, c, 1)] = word_of(l[i].y, bal, eL);
          g[word_at(r, c, 0)] = word_of(w[i].x, -bal, eW);
          g[word_at(r, c, 1)] = word_of(w[i].y, -bal, eW);
          const unsigned nl = __ballot_sync(0xffffffffu, near_max(max(exp_of(l[i].x, bal), exp_of(l[i].y, bal)), s_eL[r]));
          const unsigned nw = __ballot_sync(0xffffffffu, near_max(max(exp_of(w[i].x, -bal), exp_of(w[i].y, -bal)), s_eW[r]));
          const unsigned zl = __ballot_sync(0xffffffffu, max(exp_of(l[i].x, bal), exp_of(l[i].y, bal)) != X_ZERO);
          const unsigned zw = __ballot_sync(0xffffffffu, max(exp_of(w[i].x, -bal), exp_of(w[i].y, -bal)) != X_ZERO);
          if (lane == 0) {
            s_near[r][warp & 1] = nl;
            s_nearV[r][warp & 1] = nw;
            s_nz[r][warp & 1] = zl;
            s_nzV[r][warp & 1] = zw;
          }
        }
        __syncthreads();
        if (tid < TB) {
          EL[(int64_t)T.tile * TB + tid] = row_info(s_eL[tid], s_near[tid][0], s_near[tid][1]);
          EW[(int64_t)T.tile * TB + tid] = row_info(s_eW[tid], s_nearV[tid][0], s_nearV[tid][1]);
          ZL[(int64_t)T.tile * TB + tid] = row_nonzero(s_eL[tid], s_nz[tid][0], s_nz[tid][1]);
          ZW[(int64_t)T.tile * TB + tid] = row_nonzero(s_eW[tid], s_nzV[tid][0], s_nzV[tid][1]);
        }
      }
    }
    sched_complete(p, task);
  }

  // teardown: after a failed wait, give MMAs in flight time to land (bounded)
  if (failed || ld_volatile(&p.ctl->abort)) {
    const uint64_t t0 = globaltimer_ns();
    while (globaltimer_ns() - t0 < 2000000ull) __nanosleep(1000);
  }
  fence_before();
  __syncthreads();
  fence_after();
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u) : "memory");
}

int launch_factor_dig(const FactorParams& p, int nblocks, cudaStream_t st) {
  const size_t smem = SMEM_BYTES + 1024;   // + alignment slack
  auto kern = p.pivot ? factor_dig_kernel<true> : factor_dig_kernel<false>;
  const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return (int)e;
  kern<<<nblocks, NTHR, smem, st>>>(p);
  return (int)cudaGetLastError();
}

}  // namespace d3m
