// Persistent block-DAG factorization with a SIMT tile engine (tile edge 64).
//
// R = double: FP64 (complex128) where the digit engine's words (factor_dig.cu) do not fit; R = float: complex64 factors without tensor cores (the SIMT engine of the mixed path).
//
// Each task works on one lower tile (I, J) of L (paper Sec. II: per nonzero block a task doing
// the dense update, the dense triangular solve and the dense factorization):
//   1. S = S_in - sum_{K in segment} L_IK (D_K L_JK^T)   (S_in = K_IJ or the tile's accumulator)
//   UPDATE task: store S in the accumulator and stop.  FINAL task:
//   2a. I == J: unpivoted LDL^T of S in shared memory (scalar pivots, no conjugation),
//       breakdown check |d| >= piv_tol * max|S|; store L_JJ, D_J and L_JJ^{-1} (for the solve)
//   2b. I != J: L_IJ = S L_JJ^{-T} D_J^{-1} by a column sweep (right-looking triangular solve), eight rows a warp.
// Pivot mode (p.pivot): the diagonal tile is factored with Bunch-Kaufman symmetric pivoting
// inside the tile (1 x 1 and 2 x 2 pivots; the paper's dense kernel is sytrf, Sec. II):
// S = Lt D Lt^T with Lt = P^T L (row-permuted unit lower) and D block diagonal (d, and e for the
// sub-diagonal of each 2 x 2 block); the tile stores Lt, Lt^{-1} = L^{-1} P, d, e and the
// permutation, and the off-diagonal tiles become L_IJ = S Lt^{-T} D^{-1}, a product with the
// stored inverse; W = L D of the updates takes the 2 x 2 blocks into account.  Everything else
// (the task graph, the update order, the solve's tile products) is unchanged.
// GB300 FP64 runs at a small fraction of FP32 throughput, so the FP64 path is bound by the
// DFMA rate: a simple register-blocked 64x64 complex tile product is enough to saturate it.
#include <cuda_runtime.h>

#include "device.cuh"
#include "diag_bk.cuh"

namespace d3m {

namespace {
constexpr int TB = 64;     // tile edge
constexpr int LDS = 65;    // padded shared-memory row stride (elements)
constexpr int NTHR = 256;
}  // namespace

// Diagonal tile in pivot mode (diag_bk.cuh): stores Lt = P^T L, Lt^{-1} = L^{-1} P, d, e (2 x 2
// sub-diagonals) and the permutation; reports the smallest / largest pivot magnitude (|d|, or sqrt|det| of a
// 2 x 2 block) and the breakdown test against max|S| like the unpivoted path.
template <typename R>
__device__ __noinline__ void diag_tile_bk(const FactorParams& p, const TileTask& T, int task, typename CT<R>::C* sA,
                                          R* s_red) {
  using C = typename CT<R>::C;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  __shared__ BkShared<C> sh;
  // max |S| over the real lower triangle (breakdown scale)
  R mx = 0;
  for (int i = tid; i < TB * TB; i += NTHR) {
    const int r = i >> 6, c = i & 63;
    if (c <= r && r < T.rv) mx = fmax(mx, (R)cabs2(sA[r * LDS + c]));
  }
  for (int o = 16; o > 0; o >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  if (lane == 0) s_red[warp] = sqrt(mx);
  __syncthreads();
  R smax = 0;
  for (int w = 0; w < NTHR / 32; ++w) smax = fmax(smax, s_red[w]);
  bk_factor<R, NTHR>(sA, LDS, sh);
  // Lt = P^T L (row perm[i] of Lt = row i of L), Lt^{-1} = L^{-1} P (column perm[b] of Lt^{-1} =
  // column b of X)
  C* Lg = reinterpret_cast<C*>(p.L) + (int64_t)T.tile * TB * TB;
  C* Li = reinterpret_cast<C*>(p.Linv) + (int64_t)T.col * TB * TB;
  for (int i = tid; i < TB * TB; i += NTHR) {
    const int r = i >> 6, c = i & 63;
    const C one = CT<R>::make(c == r ? (R)1 : (R)0, 0);
    Lg[(int64_t)sh.perm[r] * TB + c] = (c < r) ? sA[r * LDS + c] : one;
    Li[(int64_t)r * TB + sh.perm[c]] = (c < r) ? sA[c * LDS + r] : one;
  }
  if (tid < TB) {
    reinterpret_cast<C*>(p.D)[(int64_t)T.col * TB + tid] = sh.d[tid];
    reinterpret_cast<C*>(p.E)[(int64_t)T.col * TB + tid] = sh.e[tid];
    p.piv[(int64_t)T.col * TB + tid] = sh.perm[tid];
  }
  if (tid < 32) {
    R amin, amax;
    bk_pivot_range<R>(sh, T.cv, amin, amax);
    if (tid == 0) {
      record_pivot_stats(p.ctl, (float)amin, (float)amax);
      if (!(amin >= (R)p.piv_tol * smax)) set_error(p.ctl, D3M_ERR_PIVOT, task);
    }
  }
}

template <typename R>
__global__ void __launch_bounds__(NTHR, 1) factor_simt_kernel(FactorParams p) {
  using C = typename CT<R>::C;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* sA = reinterpret_cast<C*>(smem_raw);       // [64][65]
  C* sB = sA + TB * LDS;                         // [64][65]
  __shared__ C s_col[TB];
  __shared__ C s_d[TB];
  __shared__ C s_tmp[TB];
  __shared__ R s_red[NTHR / 32];
  __shared__ int s_task, s_pending;
  if (threadIdx.x == 0) s_pending = -1;          // read and written by thread 0 only

  C* Lg = reinterpret_cast<C*>(p.L);
  C* Linv = reinterpret_cast<C*>(p.Linv);
  C* Dg = reinterpret_cast<C*>(p.D);
  const int tid = threadIdx.x;
  const int tx = tid & 15, ty = tid >> 4;

  for (;;) {
    const int task = sched_pop(p, &s_task, &s_pending);
    if (task < 0) break;
    const TileTask T = p.tasks[task];

    // ---------------------------------------------------------------- 1. Schur updates
    C acc[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) acc[i][j] = CT<R>::make(0, 0);
    // A thread stages entries of one column c and 16 rows.  Complex64: the next product's entries are in flight in
    // registers while this one is formed (update 11.3 -> 7.7 us a product, 4 at the FMA rate).
    constexpr int NE = TB * TB / NTHR;
    constexpr bool AHEAD = sizeof(R) == 4;
    const int c = tid & 63, rt = tid >> 6;
    C fa[AHEAD ? NE : 1], fb[AHEAD ? NE : 1], fd;
    auto fetch = [&](int e) {
      if constexpr (AHEAD) {
        const KEntry ke = p.klist[T.kl_off + e];
        const C* La = Lg + (int64_t)ke.a_tile * TB * TB + tid;
        const C* Lb = Lg + (int64_t)ke.b_tile * TB * TB + tid;
#pragma unroll
        for (int i = 0; i < NE; ++i) {
          fa[i] = ld_cg(La + i * NTHR);
          fb[i] = ld_cg(Lb + i * NTHR);
        }
        fd = ld_cg(Dg + (int64_t)ke.kcol * TB + c);
      }
    };
    if (T.nk > 0) fetch(0);
    for (int e = 0; e < T.nk; ++e) {
      const KEntry ke = p.klist[T.kl_off + e];
      const C* La = Lg + (int64_t)ke.a_tile * TB * TB;
      const C* Lb = Lg + (int64_t)ke.b_tile * TB * TB;
      const C* eK = p.E ? reinterpret_cast<const C*>(p.E) + (int64_t)ke.kcol * TB : nullptr;
      __syncthreads();
      if constexpr (!AHEAD) fd = ld_cg(Dg + (int64_t)ke.kcol * TB + c);
#pragma unroll
      for (int q = 0; q < NE; ++q) {
        const int i = tid + q * NTHR, r = rt + q * (NTHR / TB);
        sA[r * LDS + c] = AHEAD ? fa[AHEAD ? q : 0] : ld_cg(La + i);
        C w = cmul(AHEAD ? fb[AHEAD ? q : 0] : ld_cg(Lb + i), fd);    // W_JK = L_JK D_K
        if (eK) {                                               // 2 x 2 blocks of D_K
          if (c + 1 < TB) w = cfma(ld_cg(Lb + i + 1), ld_cg(eK + c), w);
          if (c > 0) w = cfma(ld_cg(Lb + i - 1), ld_cg(eK + c - 1), w);
        }
        sB[r * LDS + c] = w;
      }
      __syncthreads();
      if (e + 1 < T.nk) fetch(e + 1);
#pragma unroll 4
      for (int k = 0; k < TB; ++k) {
        C a[4], bb[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) a[i] = sA[(ty + 16 * i) * LDS + k];
#pragma unroll
        for (int j = 0; j < 4; ++j) bb[j] = sB[(tx + 16 * j) * LDS + k];
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int j = 0; j < 4; ++j) acc[i][j] = cfma(a[i], bb[j], acc[i][j]);
      }
    }
    __syncthreads();
    // the tile's accumulator lies where L_IJ ends up: its last reader, the final task, overwrites it
    C* Sa = Lg + (int64_t)T.tile * TB * TB;
    if (T.flags & TF_UPDATE) {
      // partial update: accumulator <- S_in - sum over this segment
      C kin[4][4];
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const int r = ty + 16 * i, c = tx + 16 * j;
          kin[i][j] = (T.flags & TF_S_IN) ? ld_cg(Sa + r * TB + c) : k_entry<R>(T, p.K, r, c);
        }
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) Sa[(ty + 16 * i) * TB + tx + 16 * j] = csub(kin[i][j], acc[i][j]);
      sched_complete(p, task);
      continue;
    }
    {
      C kin[4][4];
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const int r = ty + 16 * i, c = tx + 16 * j;
          kin[i][j] = (T.flags & TF_S_IN) ? ld_cg(Sa + r * TB + c) : k_entry<R>(T, p.K, r, c);
        }
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) sA[(ty + 16 * i) * LDS + tx + 16 * j] = csub(kin[i][j], acc[i][j]);
    }
    __syncthreads();

    if ((T.flags & TF_DIAG) && p.pivot) {
      // ------------------------------------------------------------ 2a'. diagonal tile, pivoted
      diag_tile_bk<R>(p, T, task, sA, s_red);
    } else if (T.flags & TF_DIAG) {
      // ------------------------------------------------------------ 2a. diagonal tile
      // max |S| over the real lower triangle; the upper triangle is zeroed to hold X^T, X = L^{-1}
      R mx = 0;
      for (int i = tid; i < TB * TB; i += NTHR) {
        const int r = i >> 6, c = i & 63;
        if (c <= r) {
          if (r < T.rv) mx = fmax(mx, (R)sqrt(cabs2(sA[r * LDS + c])));
        } else {
          sA[r * LDS + c] = CT<R>::make(0, 0);
        }
      }
      for (int o = 16; o > 0; o >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
      if ((tid & 31) == 0) s_red[tid >> 5] = mx;
      __syncthreads();
      if (tid == 0) {
        R v = 0;
        for (int w = 0; w < NTHR / 32; ++w) v = fmax(v, s_red[w]);
        s_red[0] = v;
      }
      // unpivoted LDL^T fused with the inverse of L (see the tensor-core engine): at step c,
      // l_r = S[r][c] / d_c and u_s = column c (X[c][s] above the diagonal, 1 on it, S[s][c]
      // below); rank-1 update of every (r > c, s <= r), S below / X^T above the diagonal.
      {
        const int tr = tid >> 4, tcol = tid & 15;
        for (int c = 0; c < TB; ++c) {
          if (tid < TB) {
            const C d = sA[c * LDS + c];
            const C v = sA[tid * LDS + c];
            if (tid > c) s_col[tid] = cdiv(v, d);
            s_tmp[tid] = (tid == c) ? CT<R>::make(1, 0) : v;
            if (tid == c) s_d[c] = d;
          }
          __syncthreads();
          C lr[4], us[4];
#pragma unroll
          for (int a = 0; a < 4; ++a) {
            lr[a] = s_col[tr + 16 * a];
            us[a] = s_tmp[tcol + 16 * a];
          }
#pragma unroll
          for (int a = 0; a < 4; ++a) {
            const int r = tr + 16 * a;
            if (r <= c) continue;
            C v[4];
            int off[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {          // all loads of the row first
              const int s = tcol + 16 * q;
              off[q] = (s > c) ? r * LDS + s : s * LDS + r;
              if (s <= r) v[q] = sA[off[q]];
            }
#pragma unroll
            for (int q = 0; q < 4; ++q)
              if (tcol + 16 * q <= r) sA[off[q]] = cfms(lr[a], us[q], v[q]);
          }
          __syncthreads();
          if (tid > c && tid < TB) sA[tid * LDS + c] = s_col[tid];
        }
        __syncthreads();
      }
      const R smax = s_red[0];
      // pivot checks on the real (non-padding) unknowns
      if (tid < 32) {
        R amin = (R)3.0e38, amax = 0;
        for (int c = tid; c < T.cv; c += 32) {
          const R a = (R)sqrt(cabs2(s_d[c]));
          amin = fmin(amin, a);
          amax = fmax(amax, a);
        }
        for (int o = 16; o > 0; o >>= 1) {
          amin = fmin(amin, __shfl_xor_sync(0xffffffffu, amin, o));
          amax = fmax(amax, __shfl_xor_sync(0xffffffffu, amax, o));
        }
        if (tid == 0) {
          record_pivot_stats(p.ctl, (float)amin, (float)amax);
          if (!(amin >= (R)p.piv_tol * smax)) set_error(p.ctl, D3M_ERR_PIVOT, task);
        }
      }
      // store L_JJ (unit lower), D_J, and L_JJ^{-1} (from the transposed upper storage)
      C* Lt = Lg + (int64_t)T.tile * TB * TB;
      C* Li = Linv + (int64_t)T.col * TB * TB;
      for (int i = tid; i < TB * TB; i += NTHR) {
        const int r = i >> 6, c = i & 63;
        const C one = CT<R>::make(c == r ? (R)1 : (R)0, 0);
        Lt[i] = (c < r) ? sA[r * LDS + c] : one;
        Li[i] = (c < r) ? sA[c * LDS + r] : one;
      }
      if (tid < TB) Dg[(int64_t)T.col * TB + tid] = s_d[tid];
    } else if (p.pivot) {
      // ------------------------------------------------------------ 2b'. off-diagonal, pivot mode
      // L_IJ = (S Lt_JJ^{-T}) D_J^{-1}: product with the stored inverse, then the 1 x 1 / 2 x 2
      // blocks of D_J^{-1} on the columns
      const C* Li = Linv + (int64_t)T.col * TB * TB;
      for (int i = tid; i < TB * TB; i += NTHR) {
        const int r = i >> 6, c = i & 63;
        sB[r * LDS + c] = ld_cg(Li + i);
      }
      if (tid < TB) {
        s_d[tid] = ld_cg(Dg + (int64_t)T.col * TB + tid);
        s_col[tid] = ld_cg(reinterpret_cast<const C*>(p.E) + (int64_t)T.col * TB + tid);
      }
      __syncthreads();
      C x[4][4];
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) x[i][j] = CT<R>::make(0, 0);
#pragma unroll 4
      for (int k = 0; k < TB; ++k) {
        C a[4], bb[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) a[i] = sA[(ty + 16 * i) * LDS + k];
#pragma unroll
        for (int j = 0; j < 4; ++j) bb[j] = sB[(tx + 16 * j) * LDS + k];
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int j = 0; j < 4; ++j) x[i][j] = cfma(a[i], bb[j], x[i][j]);
      }
      __syncthreads();
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) sA[(ty + 16 * i) * LDS + tx + 16 * j] = x[i][j];
      __syncthreads();
      C* Lt = Lg + (int64_t)T.tile * TB * TB;
      for (int i = tid; i < TB * TB; i += NTHR) {
        const int r = i >> 6, c = i & 63;
        const C* row = sA + r * LDS;
        C v;
        if (c + 1 < TB && (s_col[c].x != 0 || s_col[c].y != 0)) {
          // first column of a 2 x 2 block [[d_c, e], [e, d_c+1]]: [x_c x_c+1] D^{-1}
          const C e = s_col[c], d1 = s_d[c], d2 = s_d[c + 1];
          const C det = csub(cmul(d1, d2), cmul(e, e));
          v = cdiv(csub(cmul(row[c], d2), cmul(row[c + 1], e)), det);
        } else if (c > 0 && (s_col[c - 1].x != 0 || s_col[c - 1].y != 0)) {
          const C e = s_col[c - 1], d1 = s_d[c - 1], d2 = s_d[c];
          const C det = csub(cmul(d1, d2), cmul(e, e));
          v = cdiv(csub(cmul(row[c], d1), cmul(row[c - 1], e)), det);
        } else {
          v = cdiv(row[c], s_d[c]);
        }
        Lt[i] = v;
      }
    } else {
      // ------------------------------------------------------------ 2b. off-diagonal tile
      const C* Ld = Lg + (int64_t)T.diag * TB * TB;
      for (int i = tid; i < TB * TB; i += NTHR) {
        const int r = i >> 6, c = i & 63;
        sB[r * LDS + c] = ld_cg(Ld + i);
      }
      if (tid < TB) s_d[tid] = ld_cg(Dg + (int64_t)T.col * TB + tid);
      __syncthreads();
      // X L_JJ^T = S: column c of X is final once columns < c are eliminated.  The rows are independent: a warp
      // takes eight of them, two columns a lane in registers, and passes x_c around by shuffles, without barriers
      // (complex64: 75 -> 12 us a task against a sweep of the whole tile with a barrier and a division a column; 32
      // systems of m = 64 blocks: factorization 3.5 -> 1.9 ms; the same operations in the same order).
      const int lane = tid & 31, r0 = (tid >> 5) * 8;
      C x[8][2];
#pragma unroll
      for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int h = 0; h < 2; ++h) x[i][h] = sA[(r0 + i) * LDS + lane + 32 * h];
#pragma unroll
      for (int h = 0; h < 2; ++h)
#pragma unroll 4
        for (int cl = 0; cl < 32; ++cl) {
          const int c = 32 * h + cl;
          const C l0 = sB[lane * LDS + c], l1 = sB[(lane + 32) * LDS + c];
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            const C xc = CT<R>::make(__shfl_sync(0xffffffffu, x[i][h].x, cl), __shfl_sync(0xffffffffu, x[i][h].y, cl));
            if (h == 0 && lane > c) x[i][0] = cfms(xc, l0, x[i][0]);
            if (lane + 32 > c) x[i][1] = cfms(xc, l1, x[i][1]);
          }
        }
      C* Lt = Lg + (int64_t)T.tile * TB * TB;
#pragma unroll
      for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int h = 0; h < 2; ++h) Lt[(r0 + i) * TB + lane + 32 * h] = cdiv(x[i][h], s_d[lane + 32 * h]);
    }
    sched_complete(p, task);
  }
}

int launch_factor_simt(const FactorParams& p, bool fp64, int nblocks, cudaStream_t st) {
  const size_t smem = (fp64 ? sizeof(double2) : sizeof(float2)) * 2 * TB * LDS;
  cudaError_t e;
  if (fp64) {
    e = cudaFuncSetAttribute(factor_simt_kernel<double>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return (int)e;
    factor_simt_kernel<double><<<nblocks, NTHR, smem, st>>>(p);
  } else {
    e = cudaFuncSetAttribute(factor_simt_kernel<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return (int)e;
    factor_simt_kernel<float><<<nblocks, NTHR, smem, st>>>(p);
  }
  return (int)cudaGetLastError();
}

}  // namespace d3m
