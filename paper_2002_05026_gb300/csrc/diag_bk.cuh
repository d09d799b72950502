// Bunch-Kaufman LDL^T of one 64 x 64 diagonal tile in shared memory, with the inverse of L (the pivoted
// variant of the engines' diagonal tasks; the paper's dense kernel is sytrf, Sec. II).
//
// Pivots inside the tile, alpha = (1 + sqrt(17)) / 8, magnitudes |Re| + |Im|:
//   lam = max_{i > k} |S_ik| (row r); |S_kk| >= alpha lam -> 1 x 1 at k;
//   else sigma = max_{j != r} |S_rj| over the remaining matrix;
//        |S_kk| sigma >= alpha lam^2 -> 1 x 1 at k;  |S_rr| >= alpha sigma -> swap k, r, 1 x 1;
//        else swap k + 1, r and take the 2 x 2 pivot on (k, k + 1).
// Swaps are symmetric interchanges of the remaining matrix and of the rows of L computed so far.
//
// Bound by the chain of 64 pivots and, in FP64, by the FP64 pipe, where an instruction of a warp holds its SM
// partition for 64 cycles whatever its lanes do.  So one warp searches a column (two entries a lane,
// integer reductions on the magnitudes' bits, no block barrier inside a search); a trailing update packs
// two rows, a short and a long one, into the lanes of a warp; and the inverse is a rank-1 update per
// column over all threads instead of one thread per column.  FP64 tile task: 0.81 -> 0.24 ms.
#pragma once
#include "device.cuh"

namespace d3m {

constexpr int BKN = 64;                          // tile edge

template <typename C>
struct BkShared {
  C u1[BKN], u2[BKN], l1[BKN], l2[BKN];          // pivot columns before and after the division
  C d[BKN], e[BKN];                              // D: diagonal, sub-diagonal of the 2 x 2 blocks
  int perm[BKN];
  int sel[3];                                    // step size, index swapped with r (or -1), r
};

__device__ __forceinline__ double bk_abs1(double2 z) { return fabs(z.x) + fabs(z.y); }
__device__ __forceinline__ float bk_abs1(float2 z) { return fabsf(z.x) + fabsf(z.y); }

// Largest of the non-negative v1 (index i1 = lane) and v2 (index lane + 32) of a warp, negative = no
// candidate; ties to the lowest index.  Returns the index (-1: none) and the value in v.
__device__ __forceinline__ int bk_argmax(double v1, double v2, int lane, double& v) {
  const bool second = v2 > v1;
  const double b = second ? v2 : v1;
  const int i = lane + (second ? 32 : 0);
  const bool ok = b >= 0.0;
  const unsigned hi = ok ? (unsigned)__double2hiint(b) : 0u, lo = ok ? (unsigned)__double2loint(b) : 0u;
  const unsigned mh = __reduce_max_sync(0xffffffffu, hi);
  const unsigned ml = __reduce_max_sync(0xffffffffu, ok && hi == mh ? lo : 0u);
  const unsigned mi = __reduce_min_sync(0xffffffffu, ok && hi == mh && lo == ml ? (unsigned)i : 0xffffu);
  v = __hiloint2double((int)mh, (int)ml);
  return mi == 0xffffu ? -1 : (int)mi;
}
__device__ __forceinline__ int bk_argmax(float v1, float v2, int lane, float& v) {
  const bool second = v2 > v1;
  const float b = second ? v2 : v1;
  const bool ok = b >= 0.f;
  const unsigned m = __reduce_max_sync(0xffffffffu, ok ? __float_as_uint(b) : 0u);
  const unsigned mi =
      __reduce_min_sync(0xffffffffu, ok && __float_as_uint(b) == m ? (unsigned)(lane + (second ? 32 : 0)) : 0xffffu);
  v = __uint_as_float(m);
  return mi == 0xffffu ? -1 : (int)mi;
}

// All NT threads call.  sA (row stride lds): the tile, lower triangle in; out: L strictly below the diagonal
// and X = L^{-1} transposed strictly above it (sA[c][r] = X[r][c]).  sh.d, sh.e, sh.perm: D and the order.
template <typename R, int NT>
__device__ __forceinline__ void bk_factor(typename CT<R>::C* sA, int lds, BkShared<typename CT<R>::C>& sh) {
  using C = typename CT<R>::C;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  constexpr R ALPHA = (R)0.6403882032022076;     // (1 + sqrt(17)) / 8
  if (tid < BKN) {
    sh.perm[tid] = tid;
    sh.e[tid] = CT<R>::make(0, 0);
  }
  int k = 0;
  while (k < BKN) {
    __syncthreads();
    if (warp == 0) {
      R lam, sigma;
      const R v1 = lane > k ? bk_abs1(sA[lane * lds + k]) : (R)-1;
      const R v2 = lane + 32 > k ? bk_abs1(sA[(lane + 32) * lds + k]) : (R)-1;
      int r = bk_argmax(v1, v2, lane, lam);
      if (r < 0) {
        r = k;
        lam = 0;
      }
      const R akk = bk_abs1(sA[k * lds + k]);
      int step = 1, sw = -1;
      if (!(akk >= ALPHA * lam) && lam > 0) {
        auto row = [&](int t) -> R { return (t >= k && t != r) ? bk_abs1(r >= t ? sA[r * lds + t] : sA[t * lds + r]) : (R)-1; };
        if (bk_argmax(row(lane), row(lane + 32), lane, sigma) < 0) sigma = 0;
        if (akk * sigma >= ALPHA * lam * lam) {
        } else if (bk_abs1(sA[r * lds + r]) >= ALPHA * sigma) {
          sw = k;
        } else {
          sw = k + 1;
          step = 2;
        }
      }
      if (lane == 0) {
        sh.sel[0] = step;
        sh.sel[1] = sw;
        sh.sel[2] = r;
      }
    }
    __syncthreads();
    const int step = sh.sel[0], sw = sh.sel[1], r = sh.sel[2];
    // symmetric interchange of sw and r (sw < r unless sw == r)
    if (sw >= 0 && sw != r) {
      const int a = sw, b = r;
      if (tid < BKN) {
        const int t = tid;
        C *p = nullptr, *q = nullptr;
        if (t == a) {                                      // diagonal entries
          p = sA + a * lds + a;
          q = sA + b * lds + b;
        } else if (t < a) {                                // rows a and b, left of a (L so far, then k <= t < a)
          p = sA + a * lds + t;
          q = sA + b * lds + t;
        } else if (t < b) {                                // column a below a <-> row b left of b
          p = sA + t * lds + a;
          q = sA + b * lds + t;
        } else if (t > b) {                                // column a <-> column b below b
          p = sA + t * lds + a;
          q = sA + t * lds + b;
        }
        if (p) {
          const C v = *p;
          *p = *q;
          *q = v;
        }
        if (t == 0) {
          const int pv = sh.perm[a];
          sh.perm[a] = sh.perm[b];
          sh.perm[b] = pv;
        }
      }
      __syncthreads();
    }
    const int n0 = k + step;                               // first row of the remaining matrix
    if (tid < BKN) {
      if (step == 1) {
        const C d = sA[k * lds + k], v = sA[tid * lds + k];
        sh.u1[tid] = v;
        if (tid > k) sh.l1[tid] = cdiv(v, d);
        if (tid == k) sh.d[k] = d;
      } else {
        // 2 x 2 pivot D_k = [[a11, a21], [a21, a22]]: [l1 l2] = [c1 c2] D_k^{-1}
        const C a11 = sA[k * lds + k], a21 = sA[(k + 1) * lds + k], a22 = sA[(k + 1) * lds + k + 1];
        const C det = csub(cmul(a11, a22), cmul(a21, a21));
        const C c1 = tid >= n0 ? sA[tid * lds + k] : CT<R>::make(0, 0);
        const C c2 = tid >= n0 ? sA[tid * lds + k + 1] : CT<R>::make(0, 0);
        sh.u1[tid] = c1;
        sh.u2[tid] = c2;
        sh.l1[tid] = cdiv(csub(cmul(c1, a22), cmul(c2, a21)), det);
        sh.l2[tid] = cdiv(csub(cmul(c2, a11), cmul(c1, a21)), det);
        if (tid == k) {
          sh.d[k] = a11;
          sh.d[k + 1] = a22;
          sh.e[k] = a21;
        }
      }
    }
    __syncthreads();
    // the columns of L; trailing update S_rs -= l_r u_s, n0 <= s <= r, rows paired short with long
    if (tid >= n0 && tid < BKN) {
      sA[tid * lds + k] = sh.l1[tid];
      if (step == 2) sA[tid * lds + k + 1] = sh.l2[tid];
    }
    if (step == 2 && tid == 0) sA[(k + 1) * lds + k] = CT<R>::make(0, 0);   // L is unit lower inside the block
    const int m = BKN - n0;
    for (int q = warp; q < (m + 1) / 2; q += NT / 32) {
      const int ra = n0 + q, rb = BKN - 1 - q;             // lengths q + 1 and m - q
      const int len = ra == rb ? q + 1 : m + 1;
      for (int l = lane; l < len; l += 32) {
        const int rr = l <= q ? ra : rb, ss = n0 + (l <= q ? l : l - q - 1);
        C v = cfms(sh.l1[rr], sh.u1[ss], sA[rr * lds + ss]);
        if (step == 2) v = cfms(sh.l2[rr], sh.u2[ss], v);
        sA[rr * lds + ss] = v;
      }
    }
    k = n0;
  }
  __syncthreads();
  // X = L^{-1}, transposed above the diagonal: X[r][s] -= L[r][c] X[c][s] for c = 0, 1, ..., r > c >= s
  // (X[c][c] = 1; X[r][c] starts at 0, so it needs no zeroed storage)
  for (int c = 0; c + 1 < BKN; ++c) {
    const int rows = BKN - 1 - c, tot = rows * (c + 1);
    for (int i = tid; i < tot; i += NT) {
      const int rr = c + 1 + i % rows, s = i / rows;
      const C l = sA[rr * lds + c];
      C* x = sA + s * lds + rr;
      *x = s == c ? CT<R>::make(-l.x, -l.y) : cfms(l, sA[s * lds + c], *x);
    }
    __syncthreads();
  }
}

// Pivot magnitudes (|d| of 1 x 1 pivots, sqrt|det| of 2 x 2 blocks) of the first cv unknowns: smallest and
// largest, by one warp.
template <typename R>
__device__ __forceinline__ void bk_pivot_range(const BkShared<typename CT<R>::C>& sh, int cv, R& amin, R& amax) {
  const int lane = threadIdx.x & 31;
  amin = (R)3.0e38;
  amax = 0;
  for (int c = lane; c < cv; c += 32) {
    const bool first2 = c + 1 < BKN && (sh.e[c].x != 0 || sh.e[c].y != 0);
    const bool second2 = c > 0 && (sh.e[c - 1].x != 0 || sh.e[c - 1].y != 0);
    R a;
    if (first2) {
      const auto det = csub(cmul(sh.d[c], sh.d[c + 1]), cmul(sh.e[c], sh.e[c]));
      a = (R)sqrt(sqrt(cabs2(det)));
    } else if (second2) {
      continue;
    } else {
      a = (R)sqrt(cabs2(sh.d[c]));
    }
    amin = fmin(amin, a);
    amax = fmax(amax, a);
  }
  for (int o = 16; o > 0; o >>= 1) {
    amin = fmin(amin, __shfl_xor_sync(0xffffffffu, amin, o));
    amax = fmax(amax, __shfl_xor_sync(0xffffffffu, amax, o));
  }
}

}  // namespace d3m
