// Batched dense LL^T factorisation and solve of the per-cluster systems S'_k dc_k = b_k (Eq. 13; the
// paper solves them with dense LL^T, Sec. 5.1), for clusters of uneven size, one launch per step.
//
// Storage: cluster k owns an Np_k x Np_k row-major block (Np_k = 9 n_k rounded up to the tile T) whose
// lower triangle is significant.  Padding rows and columns are zero and their diagonal is treated as 1,
// so the padded system is block diagonal with an identity block and solves to zero there.
//
// The factorised matrix is the Jacobi-scaled  S~ = D^-1/2 S D^-1/2, D = diag(S) (s_i = S_ii^-1/2), so that
// S x = b becomes S~ z = s o b, x = s o z.  Right-looking tiled algorithm with a look-ahead of one column,
// step kt:
//   panel   for every tile row i >= kt: apply step kt - 1's update to tiles (kt, kt) and (i, kt), factor
//           the diagonal tile with its inverse (redundantly in each CTA); the CTA of i = kt stores
//           L_kt,kt and L_kt,kt^-1 (for the solves), the others L_i,kt = A_i,kt L_kt,kt^-T;
//   update  for every kt + 1 < j <= i: A_i,j -= L_i,kt L_j,kt^T.
// The FP32 factor with tile 64 (the default) runs panel kt + 1 and update kt as one launch of k_step_tc, on the
// tensor cores, reading S' itself where a tile is first touched.  The other factors (FP64, tile 32, CUDA-core
// updates) copy the scaled matrix first and run the updates on a second stream, overlapping the next panel.
// FP64 factor (FP64 mode): a pivot that is not positive and finite marks the cluster as failed, and the
// LM step is rejected (lambda *= 3).  FP32 factor (mixed mode): a pivot that rounding has made vanish
// (below 2^-20 of the unit scaled diagonal; legitimate pivots of the damped system are about lambda or
// more) is raised to 2^-12 and counted -- static pivoting, as in Li & Demmel's SuperLU_DIST -- and the
// FP64 iterative refinement that follows solves the unmodified system.  A non-finite pivot fails.
//
// Solves (k_tri_push): a thread-block cluster of CTAs per camera cluster; with the inverted diagonal tiles every
// tile step is two parallel matrix-vector products.  Refinement: r = b - S x in FP64 over many CTAs (S symmetric,
// lower stored), then x += D^-1/2 (L L^T)^-1 D^-1/2 r.
#include <cooperative_groups.h>

#include <map>
#include <mutex>
#include <type_traits>

#include "stba_device.cuh"
#include "stba_internal.cuh"
#include "stba_tc.cuh"

namespace stba {

#define FULL_MASK 0xffffffffu

// default tile of the factorisation: 64 for the FP32 factor (32 is the other candidate of stba_autotune),
// 32 for the FP64 factor
int factor_tile(bool mixed) { return mixed ? 64 : 32; }

// s_i = 1 / sqrt(S_ii) (1 on padding)
template <typename Sreal>
__global__ void k_diag_scale(DevProblem P, const Sreal* S, double* scale) {
  chain_begin();
  const int k = blockIdx.y;
  if (P.sharded && !P.cluster_owned[k]) return;
  const int np = P.cluster_np[k], nk = P.cluster_n[k];
  const Sreal* Sk = S + P.S_off[k];
  double* sk = scale + P.v_off[k];
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < np; i += gridDim.x * blockDim.x) {
    double d = i < nk ? (double)Sk[(size_t)i * np + i] : 1.0;
    sk[i] = d > 0.0 ? 1.0 / sqrt(d) : 1.0;
  }
}

// L = s_i s_j S_ij (lower triangle and diagonal blocks' contents; the upper part is never read), for the
// columns [c_lo, c_hi) of the lower triangle (rows from c_lo on)
template <typename Sreal, typename F>
__global__ void k_scaled_copy(DevProblem P, const Sreal* S, const double* scale, F* L, int c_lo, int c_hi) {
  const int k = blockIdx.y;
  if (P.sharded && !P.cluster_owned[k]) return;
  const int np = P.cluster_np[k];
  const Sreal* Sk = S + P.S_off[k];
  F* Lk = L + P.S_off[k];
  const double* sk = scale + P.v_off[k];
  for (int r = c_lo + blockIdx.x; r < np; r += gridDim.x) {
    const double sr = sk[r];
    const int ce = min(r, c_hi - 1);
    for (int c = c_lo + threadIdx.x; c <= ce; c += blockDim.x)
      Lk[(size_t)r * np + c] = (F)((double)Sk[(size_t)r * np + c] * sr * sk[c]);
  }
}

// Correctly rounded reciprocal (one special-function instruction plus fix-up instead of a division).
__device__ __forceinline__ float rcp_rn(float x) { return __frcp_rn(x); }
__device__ __forceinline__ double rcp_rn(double x) { return __drcp_rn(x); }

// R consecutive elements from 16-byte aligned shared memory in one vector load where the width allows.
template <typename F, int R>
__device__ __forceinline__ void load_vec(const F* p, F (&v)[R]) {
  if constexpr (sizeof(F) == 4 && R == 4) {
    const float4 t = *reinterpret_cast<const float4*>(p);
    v[0] = t.x;
    v[1] = t.y;
    v[2] = t.z;
    v[3] = t.w;
  } else if constexpr (sizeof(F) == 8 && R == 2) {
    const double2 t = *reinterpret_cast<const double2*>(p);
    v[0] = t.x;
    v[1] = t.y;
  } else {
#pragma unroll
    for (int a = 0; a < R; ++a) v[a] = p[a];
  }
}

// Asynchronous global -> shared copies of one element (4 or 8 bytes), so that all the loads of a tile are
// in flight at once and may land at transposed positions.
template <typename F>
__device__ __forceinline__ void cp_async_elem(F* smem_dst, const F* gsrc) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(smem_dst);
  if constexpr (sizeof(F) == 4)
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(d), "l"(gsrc) : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(d), "l"(gsrc) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() {
  asm volatile("cp.async.commit_group;\n" ::: "memory");
  asm volatile("cp.async.wait_group 0;\n" ::: "memory");
}
// one 16-byte asynchronous global -> shared copy (both addresses 16-byte aligned)
__device__ __forceinline__ void cp_async16(void* smem_dst, const void* gsrc) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(smem_dst);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d), "l"(gsrc) : "memory");
}

__device__ __forceinline__ float rsqrt_w(float x) { return rsqrtf(x); }
__device__ __forceinline__ double rsqrt_w(double x) { return rsqrt(x); }

// LL^T of the 8 x 8 diagonal block at (b0, b0) of a shared-memory tile, by one thread in registers; the
// reciprocal pivots go to rinv.  Pivot rules: padding rows (global row >= nk) get 1; FP64 -- a pivot that is
// not positive and finite fails the cluster; FP32 -- a non-finite pivot fails it, and a pivot that
// rounding made vanish (< 2^-20 of the unit scaled diagonal) is raised to 2^-12 and counted (static
// pivoting; the FP64 refinement solves the unmodified system).
template <typename F, int LDA>
__device__ __forceinline__ void chol8(F (*Ad)[LDA], int b0, int row0, int nk, F* rinv, int* fail, int* boosted) {
  F d[8][8];
#pragma unroll
  for (int r = 0; r < 8; ++r)
#pragma unroll
    for (int c = 0; c < 8; ++c) d[r][c] = (c <= r) ? Ad[b0 + r][b0 + c] : F(0);
  int bad = 0, nboost = 0;
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    F pv = d[j][j];
    if (row0 + b0 + j >= nk) {
      pv = F(1);
    } else if (!isfinite(pv)) {
      bad = 1;
      pv = F(1);
    } else if (sizeof(F) == 8) {
      if (!(pv > F(0))) {
        bad = 1;
        pv = F(1);
      }
    } else if (pv < F(1.0 / 1048576)) {
      ++nboost;
      pv = F(1.0 / 4096);
    }
    const F is = rsqrt_w(pv);
    d[j][j] = pv * is;
    rinv[j] = is;
#pragma unroll
    for (int r = j + 1; r < 8; ++r) d[r][j] *= is;
#pragma unroll
    for (int c = j + 1; c < 8; ++c)
#pragma unroll
      for (int r = c; r < 8; ++r) d[r][c] -= d[r][j] * d[c][j];
  }
#pragma unroll
  for (int r = 0; r < 8; ++r)
#pragma unroll
    for (int c = 0; c <= r; ++c) Ad[b0 + r][b0 + c] = d[r][c];
  if (bad) atomicOr(fail, FAIL_PIVOT);
  if (nboost && boosted) atomicAdd(boosted, nboost);
}

// The FP64 factorisation of the block by one warp: an FP64 instruction occupies the SM's pipe for 16 cycles whether
// one lane or 32 need it, and one thread's 28 reciprocal roots, products and updates a column made chol8 the longest
// part of a panel (53 us a panel of 4 clusters of 75 cameras; 34 with this, the diagonal product on its lower cells
// only and row tiles in halves).  Lane 4 r + p holds entries (r, p) and (r, p + 4): two updates a column for the
// whole block.  The same operations on every entry as in chol8, and its pivot rules.
template <int LDA>
__device__ __forceinline__ void chol8_warp(double (*Ad)[LDA], int b0, int row0, int nk, double* rinv, int* fail) {
  const int lane = threadIdx.x & 31, r = lane >> 2, p = lane & 3;
  double d0 = p <= r ? Ad[b0 + r][b0 + p] : 0.0, d1 = p + 4 <= r ? Ad[b0 + r][b0 + p + 4] : 0.0;
  int bad = 0;
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const double col = j < 4 ? d0 : d1;
    double pv = __shfl_sync(FULL_MASK, col, 4 * j + (j & 3));
    if (row0 + b0 + j >= nk) {
      pv = 1.0;
    } else if (!(isfinite(pv) && pv > 0.0)) {
      bad = 1;
      pv = 1.0;
    }
    const double is = rsqrt_w(pv);
    // L_rj of this lane's row, and L_cj for its two columns c
    const double rj = __shfl_sync(FULL_MASK, col, (lane & ~3) | (j & 3));
    const double lr = (r == j ? pv : rj) * is;
    const double l0 = __shfl_sync(FULL_MASK, lr, 4 * p), l1 = __shfl_sync(FULL_MASK, lr, 4 * p + 16);
    if (lane == 0) rinv[j] = is;
    if (p == (j & 3) && r >= j) {
      if (j < 4) d0 = lr; else d1 = lr;
    }
    if (j < 3 && p > j) d0 -= lr * l0;
    if (p + 4 > j) d1 -= lr * l1;
  }
  if (p <= r) Ad[b0 + r][b0 + p] = d0;
  if (p + 4 <= r) Ad[b0 + r][b0 + p + 4] = d1;
  if (bad && lane == 0) atomicOr(fail, FAIL_PIVOT);
}

// the block's factorisation by warp 0 (FP32: by its first thread); called by the whole warp
template <typename F, int LDA>
__device__ __forceinline__ void chol8_warp0(F (*Ad)[LDA], int b0, int row0, int nk, F* rinv, int* fail, int* boosted) {
  if constexpr (sizeof(F) == 8)
    chol8_warp<LDA>(Ad, b0, row0, nk, rinv, fail);
  else if (threadIdx.x == 0)
    chol8<F, LDA>(Ad, b0, row0, nk, rinv, fail, boosted);
}

// ------------------------------------------------------------------------------------------------------
// Panel of tile step kt, one CTA per tile row i >= kt of a cluster (512 threads: the diagonal tile's work on
// threads 0..255, the row tile's on threads 256..511, wherever the two are independent):
//   1. fused update from step kt - 1 (kt > 0):  A_kt,kt -= L_kt,kt-1 L_kt,kt-1^T,  A_i,kt -= L_i,kt-1 L_kt,kt-1^T
//      (the trailing update of the other tiles of step kt - 1 runs concurrently in k_chol_update);
//   2. LL^T of the stacked panel [A_kt,kt; A_i,kt] in blocks of 8 columns (the diagonal tile redundantly
//      in every CTA of the step): per block one thread factors the 8 x 8 diagonal block, the block
//      column below is solved against it row by row (forward substitution), and the columns to its
//      right get the rank-8 update; rows of A_i,kt are just more rows below the diagonal, so they come
//      out as L_i,kt.  The CTA of i = kt stores L_kt,kt, the others L_i,kt.
// Dynamic shared memory: Ad, Ax (T x (T + 1)) and two T x LDV buffers for the transposed tiles of the
// fused update.
constexpr int PANEL_THREADS = 512;

template <typename F, int T>
struct PanelLayout {
  static constexpr int LDA = T + 1;
  static constexpr int LDV = T + (sizeof(F) == 4 ? 4 : 2);   // 16-byte rows for vector loads
  static constexpr size_t bytes = sizeof(F) * (2 * (size_t)T * LDA + 2 * (size_t)T * LDV);
};

template <typename F, int T>
__global__ void __launch_bounds__(PANEL_THREADS) k_chol_panel(F* L, F* Ldiag, DevProblem P, const int2* items, int kt,
                                                    int* fail_flags, int* boosted) {
  using PL = PanelLayout<F, T>;
  constexpr int R = T / 16, LDA = PL::LDA, LDV = PL::LDV, NB = T / 8;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  F(*Ad)[LDA] = reinterpret_cast<F(*)[LDA]>(smem_raw);
  F(*Ax)[LDA] = Ad + T;
  F* bufV = reinterpret_cast<F*>(Ax + T);
  F(*LkT)[LDV] = reinterpret_cast<F(*)[LDV]>(bufV);
  F(*LiT)[LDV] = LkT + T;
  __shared__ F rinv2[2][8];   // reciprocal pivots of block b in rinv2[b & 1]
  const int2 it = items[blockIdx.x];
  const int k = it.x, i = it.y & 0xffff, part = it.y >> 16;   // part: 0 the whole row tile, 1 or 2 its upper or lower half
  const bool diag = (i == kt);
  const int x0 = part == 2 ? T / 2 : 0, xrows = diag ? 0 : part ? T / 2 : T;   // rows of the row tile in this CTA
  const int np = P.cluster_np[k], nk = P.cluster_n[k];
  F* A = L + P.S_off[k];
  const int tid = threadIdx.x;
  // R x R cells of a product: threads 0..255 take the diagonal tile's lower ones, threads 256..511 the row tile's
  const int half = tid >> 8, nci = xrows / R;
  int bi = 0, bj = 0;
  bool cell_act;
  if (half == 0) {
    while ((bi + 1) * (bi + 2) / 2 <= tid) ++bi;
    bj = tid - bi * (bi + 1) / 2;
    cell_act = bi < 16;
  } else {
    bi = nci ? (tid & 255) % nci : 0;
    bj = nci ? (tid & 255) / nci : 16;
    cell_act = bj < 16;
  }
  const size_t base_kk = (size_t)(kt * T) * np + kt * T;
  const size_t base_ik = (size_t)(i * T + x0) * np + kt * T;
  // 1. loads; the upper part of the diagonal tile is never stored, so it is set to zero
  for (int idx = tid; idx < T * T; idx += PANEL_THREADS) {
    const int r = idx / T, c = idx - (idx / T) * T;
    if (c <= r)
      cp_async_elem(&Ad[r][c], A + base_kk + (size_t)r * np + c);
    else
      Ad[r][c] = F(0);
    if (r < xrows) cp_async_elem(&Ax[r][c], A + base_ik + (size_t)r * np + c);
    if (kt > 0) {
      cp_async_elem(&LkT[c][r], A + base_kk - T + (size_t)r * np + c);
      if (r < xrows) cp_async_elem(&LiT[c][r], A + base_ik - T + (size_t)r * np + c);
    }
  }
  cp_async_wait_all();
  __syncthreads();
  if (kt > 0) {
    // half 0: A_kt,kt -= L_kt,kt-1 L_kt,kt-1^T (lower part); half 1: A_i,kt -= L_i,kt-1 L_kt,kt-1^T
    if (cell_act) {
      F acc[R][R];
#pragma unroll
      for (int a = 0; a < R; ++a)
#pragma unroll
        for (int b = 0; b < R; ++b) acc[a][b] = F(0);
      F(*Lr)[LDV] = half ? LiT : LkT;
#pragma unroll 4
      for (int m = 0; m < T; ++m) {
        F lr[R], lc[R];
        load_vec<F, R>(&Lr[m][bi * R], lr);
        load_vec<F, R>(&LkT[m][bj * R], lc);
#pragma unroll
        for (int a = 0; a < R; ++a)
#pragma unroll
          for (int b = 0; b < R; ++b) acc[a][b] += lr[a] * lc[b];
      }
#pragma unroll
      for (int a = 0; a < R; ++a)
#pragma unroll
        for (int b = 0; b < R; ++b) {
          const int r = bi * R + a, c = bj * R + b;
          if (half)
            Ax[r][c] -= acc[a][b];
          else if (c <= r)
            Ad[r][c] -= acc[a][b];
        }
    }
    __syncthreads();
  }
  // 2. blocked LL^T of the stacked panel.  Per block b: the rows below are solved against L_bb; then warp 0
  //    applies block b's rank-8 update to the next 8 x 8 diagonal block and lane 0 factors it, while warps
  //    1..7 apply the update to the rest of the diagonal tile and warps 8..15 to the row tile (look-ahead
  //    of one block).
  if (tid < 32) chol8_warp0<F, LDA>(Ad, 0, kt * T, nk, rinv2[0], fail_flags + k, diag ? boosted : nullptr);
  __syncthreads();
  for (int b = 0; b < NB; ++b) {
    const int b0 = 8 * b;
    const F* rinv = rinv2[b & 1];
    // block column below the diagonal block: L_rb L_bb^T = A_rb, one row per thread (Ad rows, then Ax rows)
    const int rows_d = T - b0 - 8;
    const int rows_tot = rows_d + xrows;
    if (tid < rows_tot) {
      F* row = (tid < rows_d) ? &Ad[b0 + 8 + tid][0] : &Ax[tid - rows_d][0];
      F o8[8];
#pragma unroll
      for (int c = 0; c < 8; ++c) {
        F s = row[b0 + c];
#pragma unroll
        for (int t = 0; t < c; ++t) s -= o8[t] * Ad[b0 + c][b0 + t];
        o8[c] = s * rinv[c];
      }
#pragma unroll
      for (int c = 0; c < 8; ++c) row[b0 + c] = o8[c];
    }
    __syncthreads();
    if (b + 1 == NB) break;
    const int n0 = b0 + 8;   // first column of the next block
    if (tid < 32) {
      // next diagonal block: entries (r, c), n0 <= c <= r < n0 + 8 (36 of them)
      for (int e = tid; e < 36; e += 32) {
        int rr = 0;
        while ((rr + 1) * (rr + 2) / 2 <= e) ++rr;
        const int cc = e - rr * (rr + 1) / 2;
        F s = F(0);
#pragma unroll
        for (int t = 0; t < 8; ++t) s += Ad[n0 + rr][b0 + t] * Ad[n0 + cc][b0 + t];
        Ad[n0 + rr][n0 + cc] -= s;
      }
      __syncwarp();
      chol8_warp0<F, LDA>(Ad, n0, kt * T, nk, rinv2[(b + 1) & 1], fail_flags + k, diag ? boosted : nullptr);
    } else {
      // rank-8 update of the other columns right of the block, register-blocked R x R cells: warps 1..7
      // take the diagonal tile's cells, warps 8..15 the row tile's
      const bool xpart = tid >= 256;
      for (int cell = xpart ? tid - 256 : tid - 32; cell < (xpart ? 16 * nci : 256); cell += xpart ? 256 : 224) {
        const int ci = xpart ? cell % nci : cell & 15, cj = xpart ? cell / nci : cell >> 4;
        const int c0 = cj * R, r0 = ci * R;
        if (c0 + R <= n0) continue;
        F lc[R][8];
#pragma unroll
        for (int cc = 0; cc < R; ++cc)
#pragma unroll
          for (int t = 0; t < 8; ++t) lc[cc][t] = Ad[c0 + cc][b0 + t];
        if (!xpart && cj <= ci && r0 + R > n0) {
#pragma unroll
          for (int a = 0; a < R; ++a) {
            F lr[8];
#pragma unroll
            for (int t = 0; t < 8; ++t) lr[t] = Ad[r0 + a][b0 + t];
#pragma unroll
            for (int cc = 0; cc < R; ++cc) {
              const int r = r0 + a, c = c0 + cc;
              if (c <= r && c >= n0 && r >= n0 + 8) {
                F s = F(0);
#pragma unroll
                for (int t = 0; t < 8; ++t) s += lr[t] * lc[cc][t];
                Ad[r][c] -= s;
              }
            }
          }
        }
        if (xpart) {
#pragma unroll
          for (int a = 0; a < R; ++a) {
            F xr[8];
#pragma unroll
            for (int t = 0; t < 8; ++t) xr[t] = Ax[r0 + a][b0 + t];
#pragma unroll
            for (int cc = 0; cc < R; ++cc) {
              const int c = c0 + cc;
              if (c >= n0) {
                F s = F(0);
#pragma unroll
                for (int t = 0; t < 8; ++t) s += xr[t] * lc[cc][t];
                Ax[r0 + a][c] -= s;
              }
            }
          }
        }
      }
    }
    __syncthreads();
  }
  // 3. outputs.  L_kk goes to its own buffer: later CTAs of this step may still be loading A_kk from L.
  if (diag) {
    F* Lkk = Ldiag + (size_t)P.v_off[k] * T + (size_t)kt * T * T;
    for (int idx = tid; idx < T * T; idx += PANEL_THREADS) {
      const int r = idx / T, c = idx - (idx / T) * T;
      Lkk[idx] = (c <= r) ? Ad[r][c] : F(0);
    }
    return;
  }
  for (int idx = tid; idx < xrows * T; idx += PANEL_THREADS) {
    const int r = idx / T, c = idx - (idx / T) * T;
    A[base_ik + (size_t)r * np + c] = Ax[r][c];
  }
}

// Inverse Y of a lower-triangular T x T tile D in shared memory (Y zeroed, D's upper part zero, both visible
// to every thread), by recursive doubling, 256 threads: the inverses of the 8 x 8 diagonal blocks by forward
// substitution (8 threads per block), then for h = 8, 16, .. T/2 the off-diagonal block of every 2h x 2h
// diagonal block, Y21 = -Y22 (L21 Y11), as two parallel products (Z: T * T / 2 scratch).  Ends synchronised.
template <typename F, int T>
__device__ __forceinline__ void tile_inverse(const F (*D)[T + 1], F (*Y)[T + 1], F* Z) {
  const int tid = threadIdx.x;
  if (tid < T) {   // column j of the inverse of diagonal block blk
    const int blk = tid >> 3, j = tid & 7, b0 = 8 * blk;
    F y[8];
#pragma unroll
    for (int r = 0; r < 8; ++r) {
      F s = (r == j) ? F(1) : F(0);
#pragma unroll
      for (int m = 0; m < r; ++m) s -= D[b0 + r][b0 + m] * y[m];
      y[r] = (r < j) ? F(0) : s / D[b0 + r][b0 + r];
    }
#pragma unroll
    for (int r = 0; r < 8; ++r) Y[b0 + r][b0 + j] = y[r];
  }
  __syncthreads();
  for (int h = 8; h < T; h *= 2) {
    const int n_out = T * h / 2;   // (T / 2h) pairs x h x h
    for (int e = tid; e < n_out; e += 256) {
      const int p = e / (h * h), rr = (e / h) % h, cc = e % h;
      const int r2 = (2 * p + 1) * h + rr, c1 = 2 * p * h + cc;
      F s = F(0);
      for (int q = cc; q < h; ++q) s += D[r2][2 * p * h + q] * Y[2 * p * h + q][c1];
      Z[e] = s;   // (L21 Y11)[rr][cc]
    }
    __syncthreads();
    for (int e = tid; e < n_out; e += 256) {
      const int p = e / (h * h), rr = (e / h) % h, cc = e % h;
      const int r2 = (2 * p + 1) * h + rr, c1 = 2 * p * h + cc;
      F s = F(0);
      for (int q = 0; q <= rr; ++q) s += Y[r2][(2 * p + 1) * h + q] * Z[p * h * h + q * h + cc];
      Y[r2][c1] = -s;
    }
    __syncthreads();
  }
}

// Inverse Y of every diagonal tile of the factor (for the solves), one CTA per tile (tile_inverse).  Writes
// Y row-major and its transpose at offset v_total * T.
template <typename F, int T>
__global__ void __launch_bounds__(256) k_diag_inverse(const F* Ldiag, F* Dinv, DevProblem P, const int2* items,
                                                      int64_t v_total) {
  __shared__ F D[T][T + 1];
  __shared__ F Y[T][T + 1];
  __shared__ F Z[T * T / 2];
  const int2 it = items[blockIdx.x];
  const int k = it.x, t = it.y;
  const F* Lkk = Ldiag + (size_t)P.v_off[k] * T + (size_t)t * T * T;
  const int tid = threadIdx.x;
  for (int idx = tid; idx < T * T; idx += 256) {
    const int r = idx / T, c = idx - (idx / T) * T;
    D[r][c] = (c <= r) ? Lkk[idx] : F(0);
    Y[r][c] = F(0);
  }
  __syncthreads();
  tile_inverse<F, T>(D, Y, Z);
  F* Di = Dinv + (size_t)P.v_off[k] * T + (size_t)t * T * T;
  F* DiT = Di + v_total * T;
  for (int idx = tid; idx < T * T; idx += 256) {
    const int r = idx / T, c = idx - (idx / T) * T;
    Di[idx] = Y[r][c];
    DiT[idx] = Y[c][r];
  }
}

// ------------------------------------------------------------------------------------------------------
// Split panel of tile step kt (the FP32 factor with T = 64): the diagonal tile is factored once per cluster,
// the tiles below it by a product with its inverse, so that a step's critical path is two short kernels.
//
// k_chol_diag, one CTA per cluster with a tile step kt:  A_kt,kt -= L_kt,kt-1 L_kt,kt-1^T (step kt - 1's
// update of the diagonal tile), LL^T of the tile in blocks of 8 columns (as the panel, 64 rows), and its
// inverse Y = L_kt,kt^-1 (tile_inverse), written to Dinv (row-major) and its transpose (for the solves and
// for k_chol_trsm).  Pivot rules as in chol8.
// LL^T of a T x T diagonal tile Ad (lower part; upper part zero) in shared memory, in place, 256 threads, in
// blocks of 8 columns: per block one thread factors the 8 x 8 diagonal block (chol8), the rows below are
// solved against it, and the columns to its right get the rank-8 update, warp 0 updating and factoring the
// next diagonal block meanwhile (one block of look-ahead).  row0: global row of the tile's first row (pivot
// rules of chol8 for padding rows); fail, boosted as in chol8.  Ends synchronised.
template <typename F, int T>
__device__ __forceinline__ void factor_diag_tile(F (*Ad)[T + 1], F (*rinv2)[8], int row0, int nk, int* fail,
                                                 int* boosted) {
  constexpr int R = T / 16, LDA = T + 1, NB = T / 8;
  const int tid = threadIdx.x;
  if (tid < 32) chol8_warp0<F, LDA>(Ad, 0, row0, nk, rinv2[0], fail, boosted);
  __syncthreads();
  for (int b = 0; b < NB; ++b) {
    const int b0 = 8 * b;
    const F* rinv = rinv2[b & 1];
    const int rows_d = T - b0 - 8;
    if (tid < rows_d) {
      F* row = &Ad[b0 + 8 + tid][0];
      F o8[8];
#pragma unroll
      for (int c = 0; c < 8; ++c) {
        F s = row[b0 + c];
#pragma unroll
        for (int t = 0; t < c; ++t) s -= o8[t] * Ad[b0 + c][b0 + t];
        o8[c] = s * rinv[c];
      }
#pragma unroll
      for (int c = 0; c < 8; ++c) row[b0 + c] = o8[c];
    }
    __syncthreads();
    if (b + 1 == NB) break;
    const int n0 = b0 + 8;
    if (tid < 32) {
      for (int e = tid; e < 36; e += 32) {
        int rr = 0;
        while ((rr + 1) * (rr + 2) / 2 <= e) ++rr;
        const int cc = e - rr * (rr + 1) / 2;
        F s = F(0);
#pragma unroll
        for (int t = 0; t < 8; ++t) s += Ad[n0 + rr][b0 + t] * Ad[n0 + cc][b0 + t];
        Ad[n0 + rr][n0 + cc] -= s;
      }
      __syncwarp();
      chol8_warp0<F, LDA>(Ad, n0, row0, nk, rinv2[(b + 1) & 1], fail, boosted);
    } else {
      for (int cell = tid - 32; cell < 256; cell += 224) {
        const int ci = cell & 15, cj = cell >> 4;
        const int c0 = cj * R, r0 = ci * R;
        if (c0 + R <= n0 || cj > ci || r0 + R <= n0 + 8) continue;
        F lc[R][8];
#pragma unroll
        for (int cc = 0; cc < R; ++cc)
#pragma unroll
          for (int t = 0; t < 8; ++t) lc[cc][t] = Ad[c0 + cc][b0 + t];
#pragma unroll
        for (int a = 0; a < R; ++a) {
          F lr[8];
#pragma unroll
          for (int t = 0; t < 8; ++t) lr[t] = Ad[r0 + a][b0 + t];
#pragma unroll
          for (int cc = 0; cc < R; ++cc) {
            const int r = r0 + a, c = c0 + cc;
            if (c <= r && c >= n0 && r >= n0 + 8) {
              F s = F(0);
#pragma unroll
              for (int t = 0; t < 8; ++t) s += lr[t] * lc[cc][t];
              Ad[r][c] -= s;
            }
          }
        }
      }
    }
    __syncthreads();
  }
}

template <typename F, int T>
struct DiagLayout {
  static constexpr int LDA = T + 1;
  static constexpr int LDV = T + (sizeof(F) == 4 ? 4 : 2);
  static constexpr size_t bytes = sizeof(F) * (2 * (size_t)T * LDA + (size_t)T * LDV + (size_t)T * T / 2);
};

template <typename F, int T>
__global__ void __launch_bounds__(256) k_chol_diag(const F* L, F* Dinv, DevProblem P, const int2* items, int kt,
                                                   int* fail_flags, int* boosted, int64_t v_total) {
  using DL = DiagLayout<F, T>;
  constexpr int R = T / 16, LDA = DL::LDA, LDV = DL::LDV;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  F(*Ad)[LDA] = reinterpret_cast<F(*)[LDA]>(smem_raw);
  F(*Y)[LDA] = Ad + T;
  F(*LkT)[LDV] = reinterpret_cast<F(*)[LDV]>(Y + T);
  F* Z = reinterpret_cast<F*>(LkT + T);
  __shared__ F rinv2[2][8];
  const int k = items[blockIdx.x].x;
  const int np = P.cluster_np[k], nk = P.cluster_n[k];
  const F* A = L + P.S_off[k];
  const int tid = threadIdx.x;
  const int bi = tid & 15, bj = tid >> 4;
  const size_t base_kk = (size_t)(kt * T) * np + kt * T;
  for (int idx = tid; idx < T * T; idx += 256) {
    const int r = idx / T, c = idx - (idx / T) * T;
    if (c <= r)
      cp_async_elem(&Ad[r][c], A + base_kk + (size_t)r * np + c);
    else
      Ad[r][c] = F(0);
    Y[r][c] = F(0);
    if (kt > 0) cp_async_elem(&LkT[c][r], A + base_kk - T + (size_t)r * np + c);
  }
  cp_async_wait_all();
  __syncthreads();
  if (kt > 0) {   // A_kk -= L_k,kt-1 L_k,kt-1^T (lower part)
    F acc[R][R];
#pragma unroll
    for (int a = 0; a < R; ++a)
#pragma unroll
      for (int b = 0; b < R; ++b) acc[a][b] = F(0);
#pragma unroll 4
    for (int m = 0; m < T; ++m) {
      F lr[R], lc[R];
      load_vec<F, R>(&LkT[m][bi * R], lr);
      load_vec<F, R>(&LkT[m][bj * R], lc);
#pragma unroll
      for (int a = 0; a < R; ++a)
#pragma unroll
        for (int b = 0; b < R; ++b) acc[a][b] += lr[a] * lc[b];
    }
#pragma unroll
    for (int a = 0; a < R; ++a)
#pragma unroll
      for (int b = 0; b < R; ++b) {
        const int r = bi * R + a, c = bj * R + b;
        if (c <= r) Ad[r][c] -= acc[a][b];
      }
    __syncthreads();
  }
  factor_diag_tile<F, T>(Ad, rinv2, kt * T, nk, fail_flags + k, boosted);
  tile_inverse<F, T>(Ad, Y, Z);
  F* Di = Dinv + (size_t)P.v_off[k] * T + (size_t)kt * T * T;
  F* DiT = Di + v_total * T;
  for (int idx = tid; idx < T * T; idx += 256) {
    const int r = idx / T, c = idx - (idx / T) * T;
    Di[idx] = Y[r][c];
    DiT[idx] = Y[c][r];
  }
}

// k_chol_trsm, one CTA per tile row i > kt of a cluster with a tile step kt:
//   A_i,kt -= L_i,kt-1 L_kt,kt-1^T   (step kt - 1's update of the tile)
//   L_i,kt  = A_i,kt Y^T              (Y = L_kt,kt^-1 from k_chol_diag: the triangular solve as a product)
// both as 64 x 64 x 64 register-blocked products (4 x 4 per thread) over transposed shared-memory tiles.
template <typename F, int T>
struct TrsmLayout {
  static constexpr int LD = T + (sizeof(F) == 4 ? 4 : 2);
  static constexpr size_t bytes = sizeof(F) * 4 * (size_t)T * LD;
};

template <typename F, int T>
__global__ void __launch_bounds__(256) k_chol_trsm(F* L, const F* Dinv, DevProblem P, const int2* items, int kt,
                                                   int64_t v_total) {
  constexpr int R = T / 16, LD = TrsmLayout<F, T>::LD;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  F(*AT)[LD] = reinterpret_cast<F(*)[LD]>(smem_raw);   // A_i,kt transposed
  F(*YT)[LD] = AT + T;                                   // Y^T (row m, column c = Y[c][m])
  F(*LiT)[LD] = YT + T;                                  // L_i,kt-1 transposed
  F(*LkT)[LD] = LiT + T;                                 // L_kt,kt-1 transposed
  const int2 it = items[blockIdx.x];
  const int k = it.x, i = it.y;
  const int np = P.cluster_np[k];
  F* A = L + P.S_off[k];
  const F* DiT = Dinv + v_total * T + (size_t)P.v_off[k] * T + (size_t)kt * T * T;
  const size_t base_ik = (size_t)(i * T) * np + kt * T, base_kk = (size_t)(kt * T) * np + kt * T;
  const int tid = threadIdx.x;
  for (int idx = tid; idx < T * T; idx += 256) {
    const int r = idx / T, c = idx - (idx / T) * T;
    cp_async_elem(&AT[c][r], A + base_ik + (size_t)r * np + c);
    if (kt > 0) {
      cp_async_elem(&LiT[c][r], A + base_ik - T + (size_t)r * np + c);
      cp_async_elem(&LkT[c][r], A + base_kk - T + (size_t)r * np + c);
    }
  }
  {
    constexpr int CH = T * (int)sizeof(F) / 16;   // 16-byte chunks per row of Y^T
    for (int q = tid; q < T * CH; q += 256) {
      const int r = q / CH, c = q - (q / CH) * CH;
      cp_async16(&YT[r][c * (16 / (int)sizeof(F))], DiT + (size_t)r * T + c * (16 / (int)sizeof(F)));
    }
  }
  cp_async_wait_all();
  __syncthreads();
  const int tr = tid >> 4, tc = tid & 15;
  if (kt > 0) {
    F acc[R][R];
#pragma unroll
    for (int a = 0; a < R; ++a)
#pragma unroll
      for (int b = 0; b < R; ++b) acc[a][b] = F(0);
#pragma unroll 4
    for (int m = 0; m < T; ++m) {
      F av[R], bv[R];
      load_vec<F, R>(&LiT[m][tr * R], av);
      load_vec<F, R>(&LkT[m][tc * R], bv);
#pragma unroll
      for (int a = 0; a < R; ++a)
#pragma unroll
        for (int b = 0; b < R; ++b) acc[a][b] += av[a] * bv[b];
    }
#pragma unroll
    for (int a = 0; a < R; ++a)
#pragma unroll
      for (int b = 0; b < R; ++b) AT[tc * R + b][tr * R + a] -= acc[a][b];
    __syncthreads();
  }
  F acc[R][R];
#pragma unroll
  for (int a = 0; a < R; ++a)
#pragma unroll
    for (int b = 0; b < R; ++b) acc[a][b] = F(0);
#pragma unroll 4
  for (int m = 0; m < T; ++m) {
    F av[R], bv[R];
    load_vec<F, R>(&AT[m][tr * R], av);
    load_vec<F, R>(&YT[m][tc * R], bv);
#pragma unroll
    for (int a = 0; a < R; ++a)
#pragma unroll
      for (int b = 0; b < R; ++b) acc[a][b] += av[a] * bv[b];
  }
#pragma unroll
  for (int a = 0; a < R; ++a)
#pragma unroll
    for (int b = 0; b < R; ++b) A[base_ik + (size_t)(tr * R + a) * np + tc * R + b] = acc[a][b];
}

// A_ij -= L_i,kt L_j,kt^T on a T x T tile; 256 threads, each an (T/16) x (T/16) register block.
template <typename F, int T>
__global__ void __launch_bounds__(256) k_chol_update(F* L, DevProblem P, const int2* items, int kt) {
  constexpr int R = T / 16;
  constexpr int LD = T + (sizeof(F) == 4 ? 4 : 2);
  __shared__ __align__(16) F LiT[T][LD];
  __shared__ __align__(16) F LjT[T][LD];
  const int2 it = items[blockIdx.x];
  const int k = it.x, i = it.y >> 16, j = it.y & 0xffff;
  const int np = P.cluster_np[k];
  F* A = L + P.S_off[k];
  const size_t bi = (size_t)(i * T) * np + kt * T, bj = (size_t)(j * T) * np + kt * T;
  for (int idx = threadIdx.x; idx < T * T; idx += blockDim.x) {
    const int r = idx / T, c = idx - (idx / T) * T;
    cp_async_elem(&LiT[c][r], A + bi + (size_t)r * np + c);
    cp_async_elem(&LjT[c][r], A + bj + (size_t)r * np + c);
  }
  cp_async_wait_all();
  __syncthreads();
  const int tr = threadIdx.x >> 4, tc = threadIdx.x & 15;
  F acc[R][R];
#pragma unroll
  for (int a = 0; a < R; ++a)
#pragma unroll
    for (int b = 0; b < R; ++b) acc[a][b] = F(0);
#pragma unroll 4
  for (int kk = 0; kk < T; ++kk) {
    F av[R], bv[R];
    load_vec<F, R>(&LiT[kk][tr * R], av);
    load_vec<F, R>(&LjT[kk][tc * R], bv);
#pragma unroll
    for (int a = 0; a < R; ++a)
#pragma unroll
      for (int b = 0; b < R; ++b) acc[a][b] += av[a] * bv[b];
  }
  const size_t bij = (size_t)(i * T) * np + j * T;
#pragma unroll
  for (int a = 0; a < R; ++a)
#pragma unroll
    for (int b = 0; b < R; ++b) A[bij + (size_t)(tr * R + a) * np + tc * R + b] -= acc[a][b];
}

// ------------------------------------------------------------------------------------------------------
// Trailing update on the fifth-generation tensor cores (FP32 factor, T = 64).  One CTA per item (k, i0, j)
// updates the two tiles (i0, j) and (i0 + 1, j) of cluster k:  [A_i0,j; A_i0+1,j] -= [L_i0,kt; L_i0+1,kt] L_j,kt^T,
// one 128 x 64 x 64 product D = A B^T by tcgen05.mma (kind::tf32, FP32 accumulation in tensor memory).
// FP32 accuracy from TF32 operands: every value x is split into hi = tf32(x) and lo = tf32(x - hi), and
// D = A_hi B_lo + A_lo B_hi + A_hi B_hi (3xTF32; the dropped A_lo B_lo is below FP32 rounding), 24 MMAs
// of K = 8 issued by one thread.  The split operands were written by the panel that made the column, in the no-swizzle
// K-major core-matrix layout (stba_tc.cuh), 32 KB per tile, so that six bulk copies bring them in and no thread
// converts anything; the product goes from TMEM through shared memory, so that the updated values are
// read and written 256 contiguous bytes per row.  The waits for the copies and
// the MMAs are bounded: a CTA that gives up marks the cluster failed (the LM step is rejected), waits, bounded again,
// for what it has in flight, frees its tensor memory and returns.  When i0 + 1 is past the cluster's last tile, the
// second half of A is undefined and its rows are not written.
// Bound by L2 traffic (96 KB of operands, 64 KB of updated values per tile pair).  With operands loaded, split and
// stored by the threads the factorisation stage took 1194 us instead of 922 (13 uneven clusters), 853 instead of 707
// (one of 400 cameras); with one row per lane and 16 bytes per access on top, the L1 pipe was 71 % busy.
constexpr int TCU_THREADS = 256;
constexpr size_t TCU_SMEM = sizeof(uint32_t) * (2 * 128 * 64 + 2 * 64 * 64);   // A hi/lo, B hi/lo: 96 KB

__device__ __forceinline__ void split_store(uint32_t* hi, uint32_t* lo, int off, float4 v) {
  const uint32_t h0 = tc::to_tf32(v.x), h1 = tc::to_tf32(v.y), h2 = tc::to_tf32(v.z), h3 = tc::to_tf32(v.w);
  *reinterpret_cast<uint4*>(hi + off) = make_uint4(h0, h1, h2, h3);
  *reinterpret_cast<uint4*>(lo + off) =
      make_uint4(tc::to_tf32(v.x - __uint_as_float(h0)), tc::to_tf32(v.y - __uint_as_float(h1)),
                 tc::to_tf32(v.z - __uint_as_float(h2)), tc::to_tf32(v.w - __uint_as_float(h3)));
}

// One CTA's work in a tile step: cluster, tile row (panel) or (i0 << 16) | j (update), and the cluster's layout.
struct TileTask {
  int k, tile, np, nk;
  int64_t S_off, v_off;
};

// A step CTA's barriers (operands loaded, MMAs done) and tensor memory.
struct StepShared {
  uint64_t mbar_load, mbar;
  uint32_t taddr;
};

// A step's product accumulates in two halves of K (64 columns of tensor memory each), added in FP32: the tensor cores'
// sums are less exact than FP32 additions at the accumulator's magnitude, which each half has to bear half as often at
// half the size.  The unrefined step's distance from the exact one, with one accumulator -> with two (with FP32 panel
// updates on the CUDA cores): 500 photos, lambda 0.01, 1.15e-6 -> 9.8e-7 (1.04e-6); 150 photos 1.22e-6 -> 1.05e-6
// (1.10e-6); four accumulators 1.03e-6, but 10 % more time.
constexpr uint32_t STEP_TMEM = 128;
__device__ __forceinline__ void load_product(uint32_t taddr, float (&d)[32]) {
  float e[32];
  tc::tmem_ld32(taddr, d);
  tc::tmem_ld32(taddr + 64, e);
#pragma unroll
  for (int u = 0; u < 32; ++u) d[u] += e[u];
}

// The end of a step CTA that gave up: its copies (loads) and products (multiplied; thread 0's knowledge) end before its
// shared and tensor memory are handed back.
__device__ __forceinline__ void step_give_up(StepShared& hs, int* fail, bool loads, bool multiplied) {
  if (threadIdx.x == 0) {
    atomicOr(fail, FAIL_WAIT);
    if (loads) tc::mbar_wait_bounded(&hs.mbar_load, 0, tc::WAIT_NS);
    if (multiplied) tc::mbar_wait_bounded(&hs.mbar, 0, tc::WAIT_NS);
  }
  __syncthreads();
  if (threadIdx.x < 32) tc::tmem_dealloc(hs.taddr, STEP_TMEM);
}

// Four values of row `row`, columns col .. col + 3 of cluster k's scaled matrix, from the FP64 S' (the first touch of a
// tile reads S' itself: no scaled copy is made for the tensor-core factorisation).
__device__ __forceinline__ float4 scaled4(const double* __restrict__ Sk, const double* sk, int np, int row,
                                          int col) {
  const double2* p = reinterpret_cast<const double2*>(Sk + (size_t)row * np + col);
  const double2 a = p[0], b = p[1];
  const double sr = sk[row];
  return make_float4((float)(a.x * sr * sk[col]), (float)(a.y * sr * sk[col + 1]), (float)(b.x * sr * sk[col + 2]),
                     (float)(b.y * sr * sk[col + 3]));
}

// The split operands of a tile column: hi and lo parts of every tile, in the core-matrix layout, SPLIT_TILE words per
// tile at its row offset; written by the panel that makes the column, read by the next launch (two columns in turn).
constexpr int SPLIT_TILE = 2 * 64 * 64;
__device__ __forceinline__ uint32_t* split_tile(uint32_t* split, int64_t v_total, int64_t v_off, int tile, int kt) {
  return split + (size_t)(kt & 1) * v_total * 128 + (size_t)(v_off + tile * 64) * 128;
}

// FIRST: step 0, whose old values come from S' (every tile this kernel ever updates is in its list there).
template <bool FIRST>
__device__ __forceinline__ void update_pair_tc(uint32_t* tsm, StepShared& hs, float* L, uint32_t* split,
                                               const double* __restrict__ S, const double* scale,
                                               const TileTask& task, int kt, int* fail_flags, int64_t v_total,
                                               uint32_t wait_ns) {
  constexpr int T = 64, LDS_ = 68;   // staging rows of the product: 16-byte aligned, no bank conflicts
  uint32_t* Ah = tsm;   // 128 x 64 TF32, core-matrix layout
  uint32_t* Al = tsm + 128 * 64;
  uint32_t* Bh = tsm + 2 * 128 * 64;   // 64 x 64
  uint32_t* Bl = Bh + 64 * 64;
  float* stage = reinterpret_cast<float*>(tsm);   // over A, once the MMAs are done
  const int k = task.k, i0 = task.tile >> 16, j = task.tile & 0xffff;
  const int np = task.np;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int rows_valid = min(128, np - i0 * T);   // 64 or 128
  const uint32_t tmem = hs.taddr;
  // operands by the copy engine; the second half of A stays undefined past the last tile (its rows are not used)
  bool multiplied = false;
  if (tid == 0) {
    const bool two = rows_valid == 128;
    tc::fence_async_all();
    tc::mbar_arrive_expect(&hs.mbar_load, (two ? 6u : 4u) * 16384u);
    const uint32_t* a0 = split_tile(split, v_total, task.v_off, i0, kt);
    const uint32_t* b = split_tile(split, v_total, task.v_off, j, kt);
    tc::bulk_load(Ah, a0, 16384, &hs.mbar_load);
    tc::bulk_load(Al, a0 + 4096, 16384, &hs.mbar_load);
    tc::bulk_load(Bh, b, 16384, &hs.mbar_load);
    tc::bulk_load(Bl, b + 4096, 16384, &hs.mbar_load);
    if (two) {
      tc::bulk_load(Ah + 4096, a0 + SPLIT_TILE, 16384, &hs.mbar_load);
      tc::bulk_load(Al + 4096, a0 + SPLIT_TILE + 4096, 16384, &hs.mbar_load);
    }
    multiplied = tc::mbar_wait_bounded(&hs.mbar_load, 0, wait_ns);
    if (multiplied) {
      tc::fence_after_sync();
      constexpr uint32_t idesc = tc::idesc_tf32(128, 64);
      const uint32_t pa[3] = {tc::smem_u32(Ah), tc::smem_u32(Al), tc::smem_u32(Ah)};
      const uint32_t pb[3] = {tc::smem_u32(Bl), tc::smem_u32(Bh), tc::smem_u32(Bh)};
#pragma unroll
      for (int pass = 0; pass < 3; ++pass)
#pragma unroll
        for (int ks = 0; ks < 8; ++ks)
          tc::mma_tf32(tmem + 64 * (ks / 4), tc::smem_desc(pa[pass] + ks * 256, 128, 2048), tc::smem_desc(pb[pass] + ks * 256, 128, 2048),
                       idesc, (pass | (ks & 3)) != 0);
      tc::mma_commit(&hs.mbar);
    }
  }
  // the updated values: 16 lanes per row (256 contiguous bytes), rows 16 v + tid / 16
  const int r16 = tid >> 4, c4 = 4 * (tid & 15);
  float* dst = L + task.S_off + (size_t)(i0 * T + r16) * np + j * T + c4;
  float4 old[8];
#pragma unroll
  for (int v = 0; v < 8; ++v) {
    if (16 * v + r16 >= rows_valid) {
      old[v] = make_float4(0.f, 0.f, 0.f, 0.f);
    } else if constexpr (FIRST) {
      old[v] = scaled4(S + task.S_off, scale + task.v_off, np, i0 * T + 16 * v + r16, j * T + c4);
    } else {
      old[v] = *reinterpret_cast<const float4*>(dst + (size_t)(16 * v) * np);
    }
  }
  __syncwarp();
  // thread (lane quarter warp & 3, column half warp >> 2): row R of the product, 32 columns, to the staging rows
  const bool done = __all_sync(0xffffffffu, tc::mbar_wait_bounded(&hs.mbar, 0, wait_ns));
  if (done) {
    tc::fence_after_sync();
    float d[32];
    const int R = 32 * (warp & 3) + lane, c0 = 32 * (warp >> 2);
    load_product(tmem + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)c0, d);
#pragma unroll
    for (int v = 0; v < 8; ++v)
      *reinterpret_cast<float4*>(stage + R * LDS_ + c0 + 4 * v) = make_float4(d[4 * v], d[4 * v + 1], d[4 * v + 2], d[4 * v + 3]);
  }
  tc::fence_before_sync();
  if (!__syncthreads_and(done)) return step_give_up(hs, fail_flags + k, true, multiplied);
  if (warp == 0) tc::tmem_dealloc(tmem, STEP_TMEM);
#pragma unroll
  for (int v = 0; v < 8; ++v) {
    if (16 * v + r16 >= rows_valid) break;
    const float4 d = *reinterpret_cast<const float4*>(stage + (16 * v + r16) * LDS_ + c4);
    *reinterpret_cast<float4*>(dst + (size_t)(16 * v) * np) =
        make_float4(old[v].x - d.x, old[v].y - d.y, old[v].z - d.z, old[v].w - d.w);
  }
}

// ------------------------------------------------------------------------------------------------------
// Panel of tile step kt with the tensor-core update (FP32 factor, T = 64): one CTA per tile row i >= kt of a
// cluster works on the stacked tile [A_kt,kt; A_i,kt] (128 rows; the CTA of i = kt takes the identity as its lower
// half, whose rows then come out as L_kt,kt^-T: the inverse the solves need, at no extra step).
//   1. step kt - 1's update, [A_kt; A_i] -= [L_kt,kt-1; L_i,kt-1] L_kt,kt-1^T, is one 128 x 64 x 64 product on the
//      tensor cores (3xTF32 as update_pair_tc; B is the first half of A), the old values loaded meanwhile;
//   2. LL^T of the stack in blocks of 8 columns, left-looking: thread r < 128 owns row r.  Between two barriers warp
//      4 applies the last block's rank-8 term to the 8 x 8 diagonal block and its lane 0 factors it, while every
//      row below finishes the same block column in its registers and takes the terms of all earlier blocks off
//      the next one; between the next two barriers the rows are solved against the factored block and stored.
// The chain is the 64 pivots (about 55 cycles each in chol8_fast) plus two barriers and one 8-step substitution per
// block.  A row's operands are its own smem row (16-byte loads, 68-float rows: no bank conflicts) and the diagonal
// rows, which all lanes read at one address, so that a block moves a quarter of the shared-memory words of the
// right-looking rank-8 updates of k_chol_panel, which bound it.  The terms of a block of columns are summed from zero
// before they come off an entry (dot8): taken off one by one, they round eight times as often at the entry's
// magnitude, and the unrefined step was 1.5 times as far from the exact one (120 cameras, lambda 0.05: 1.12e-6 against
// 7.4e-7, which k_chol_panel has too), at the same time per step.
// Panel alone on an SM: about 8.5 us (loads 1.5, product 0.65, sweep 5.9; k_chol_panel took 20), beside an
// update CTA about 12.  Warps 5 .. 7 write each finished block out (factor, split operands, inverse).  One 512-thread
// CTA per SM with two tasks, so that a panel has its SM to itself, was slower (12 clusters of 83 cameras 265 us
// against 228: an SM then waits for both tasks).
constexpr int PTC_THREADS = 256;
constexpr int PTC_LD = 68;
constexpr size_t PTC_SMEM = sizeof(float) * 128 * PTC_LD + sizeof(uint32_t) * 2 * 128 * 64;   // tile, A hi / lo: 98 KB

__device__ __forceinline__ float rsqrt_normal(float x) {   // x normal and positive (pivots are >= 2^-20)
  float r;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

// LL^T of the 8 x 8 block at T (rows of PTC_LD floats), by one thread in registers; reciprocal pivots to rinv.
// The pivot rules of chol8 (FP32).
__device__ __forceinline__ void chol8_fast(float* T, int row0, int nk, float* rinv, int* fail, int* boosted) {
  float d[8][8];
#pragma unroll
  for (int r = 0; r < 8; ++r) {
    const float4 a = *reinterpret_cast<const float4*>(T + r * PTC_LD);
    d[r][0] = a.x;
    d[r][1] = a.y;
    d[r][2] = a.z;
    d[r][3] = a.w;
    if (r >= 4) {
      const float4 b = *reinterpret_cast<const float4*>(T + r * PTC_LD + 4);
      d[r][4] = b.x;
      d[r][5] = b.y;
      d[r][6] = b.z;
      d[r][7] = b.w;
    }
  }
  int bad = 0, nboost = 0;
  float ri[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    float pv = d[j][j];
    const bool pad = row0 + j >= nk, fin = isfinite(pv), low = pv < 1.f / 1048576;
    bad |= !pad && !fin;
    nboost += !pad && fin && low;
    pv = (pad || !fin) ? 1.f : (low ? 1.f / 4096 : pv);
    const float is = rsqrt_normal(pv);
    d[j][j] = pv * is;
    ri[j] = is;
#pragma unroll
    for (int r = j + 1; r < 8; ++r) d[r][j] *= is;
#pragma unroll
    for (int c = j + 1; c < 8; ++c)
#pragma unroll
      for (int r = c; r < 8; ++r) d[r][c] -= d[r][j] * d[c][j];
  }
#pragma unroll
  for (int r = 1; r < 8; ++r) {
    *reinterpret_cast<float4*>(T + r * PTC_LD) =
        make_float4(d[r][0], r > 1 ? d[r][1] : 0.f, r > 2 ? d[r][2] : 0.f, r > 3 ? d[r][3] : 0.f);
    if (r > 4)
      *reinterpret_cast<float4*>(T + r * PTC_LD + 4) =
          make_float4(d[r][4], r > 5 ? d[r][5] : 0.f, r > 6 ? d[r][6] : 0.f, 0.f);   // below the diagonal only
  }
  reinterpret_cast<float4*>(rinv)[0] = make_float4(ri[0], ri[1], ri[2], ri[3]);
  reinterpret_cast<float4*>(rinv)[1] = make_float4(ri[4], ri[5], ri[6], ri[7]);
  if (bad) atomicOr(fail, FAIL_PIVOT);
  if (nboost && boosted) atomicAdd(boosted, nboost);
}

// a.b over one block of eight columns, summed from zero: the terms of a block come off an entry with one rounding at
// the entry's magnitude, not eight
__device__ __forceinline__ float dot8(float4 a0, float4 a1, const float* b) {
  const float4 b0 = *reinterpret_cast<const float4*>(b), b1 = *reinterpret_cast<const float4*>(b + 4);
  float s = a0.x * b0.x;
  s = fmaf(a0.y, b0.y, s);
  s = fmaf(a0.z, b0.z, s);
  s = fmaf(a0.w, b0.w, s);
  s = fmaf(a1.x, b1.x, s);
  s = fmaf(a1.y, b1.y, s);
  s = fmaf(a1.z, b1.z, s);
  return fmaf(a1.w, b1.w, s);
}

__device__ __forceinline__ void panel_tc(uint32_t* psm, StepShared& hs, float* L, float* Dinv, uint32_t* split,
                                         const double* __restrict__ S, const double* scale,
                                         const TileTask& task, int kt, int* fail_flags, int* boosted, int64_t v_total,
                                         uint32_t wait_ns) {
  constexpr int T = 64, LD = PTC_LD, NB = T / 8;
  uint32_t* Ah = psm;   // 128 x 64 TF32, core-matrix layout: rows of L_kt,kt-1, then of L_i,kt-1
  uint32_t* Al = psm + 128 * 64;
  float* W = reinterpret_cast<float*>(psm + 2 * 128 * 64);   // [128][LD] the stacked tile
  __shared__ __align__(16) float rinv[8];
  const int k = task.k, i = task.tile;
  const bool diag = i == kt;
  const int np = task.np, nk = task.nk;
  float* A = L + task.S_off;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t tmem = hs.taddr;
  if (kt > 0 && tid == 0) {   // the operands by the copy engine
    tc::fence_async_all();
    tc::mbar_arrive_expect(&hs.mbar_load, (diag ? 2u : 4u) * 16384u);
    const uint32_t* a0 = split_tile(split, v_total, task.v_off, kt, kt - 1);
    tc::bulk_load(Ah, a0, 16384, &hs.mbar_load);
    tc::bulk_load(Al, a0 + 4096, 16384, &hs.mbar_load);
    if (!diag) {   // else rows 64 .. stay undefined: their product is not used
      const uint32_t* a1 = split_tile(split, v_total, task.v_off, i, kt - 1);
      tc::bulk_load(Ah + 4096, a1, 16384, &hs.mbar_load);
      tc::bulk_load(Al + 4096, a1 + 4096, 16384, &hs.mbar_load);
    }
  }
  // the stacked tile's old values: 16 lanes per row; columns 0 and 1 come from S' (no update has touched them)
  const int r16 = tid >> 4, c4 = 4 * (tid & 15);
#pragma unroll
  for (int v = 0; v < 8; ++v) {
    const int r = 16 * v + r16, grow = r < T ? kt * T + r : i * T + r - T;
    float* w = W + r * LD + c4;
    if (v >= 4 && diag) {   // the identity
      const int e = r - T - c4;
      *reinterpret_cast<float4*>(w) = make_float4(e == 0 ? 1.f : 0.f, e == 1 ? 1.f : 0.f, e == 2 ? 1.f : 0.f, e == 3 ? 1.f : 0.f);
    } else if (kt <= 1) {
      *reinterpret_cast<float4*>(w) = scaled4(S + task.S_off, scale + task.v_off, np, grow, kt * T + c4);
    } else {
      cp_async16(w, A + (size_t)grow * np + kt * T + c4);
    }
  }
  bool done = true, multiplied = false;
  if (kt > 0) {
    if (tid == 0) multiplied = tc::mbar_wait_bounded(&hs.mbar_load, 0, wait_ns);
    if (multiplied) {
      tc::fence_after_sync();
      constexpr uint32_t idesc = tc::idesc_tf32(128, 64);
      const uint32_t pa[3] = {tc::smem_u32(Ah), tc::smem_u32(Al), tc::smem_u32(Ah)};
      const uint32_t pb[3] = {tc::smem_u32(Al), tc::smem_u32(Ah), tc::smem_u32(Ah)};   // rows 0 .. 63
#pragma unroll
      for (int pass = 0; pass < 3; ++pass)
#pragma unroll
        for (int ks = 0; ks < 8; ++ks)
          tc::mma_tf32(tmem + 64 * (ks / 4), tc::smem_desc(pa[pass] + ks * 256, 128, 2048), tc::smem_desc(pb[pass] + ks * 256, 128, 2048),
                       idesc, (pass | (ks & 3)) != 0);
      tc::mma_commit(&hs.mbar);
    }
    cp_async_wait_all();
    __syncthreads();   // the old values are in place
    done = __all_sync(FULL_MASK, tc::mbar_wait_bounded(&hs.mbar, 0, wait_ns));
    if (done) {
      tc::fence_after_sync();
      float d[32];
      const int R = 32 * (warp & 3) + lane, c0 = 32 * (warp >> 2);   // a row and half of its columns
      load_product(tmem + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)c0, d);
      if (R < T || !diag) {
#pragma unroll
        for (int v = 0; v < 8; ++v) {
          float4* w = reinterpret_cast<float4*>(W + R * LD + c0 + 4 * v);
          float4 a = *w;
          a.x -= d[4 * v];
          a.y -= d[4 * v + 1];
          a.z -= d[4 * v + 2];
          a.w -= d[4 * v + 3];
          *w = a;
        }
      }
    }
    tc::fence_before_sync();
  }
  // a wait gave up: the cluster fails, the step is rejected
  if (!__syncthreads_and(done)) return step_give_up(hs, fail_flags + k, true, multiplied);
  if (warp == 0) tc::tmem_dealloc(tmem, STEP_TMEM);
  float* my = W + tid * LD;   // row threads
  float x[8], nx[8], o[8];
  float* Di = Dinv + (size_t)task.v_off * T + (size_t)kt * T * T;
  float* DiT = Di + v_total * T;
  uint32_t* Xs = diag ? nullptr : split_tile(split, v_total, task.v_off, i, kt);
  float* Xg = diag ? DiT : A + (size_t)(i * T) * np + kt * T;   // where the lower rows go
  const size_t Xld = diag ? (size_t)T : (size_t)np;
  // warps 5 .. 7: the lower rows' solved columns n0 .. n0 + 7 from shared memory to the factor (or the inverse) and
  // to the split operands
  auto store_block = [&](int n0) {
    for (int c = tid - 160; c < 128; c += 96) {
      const int r = c & 63, col = n0 + 4 * (c >> 6);
      const float4 v = *reinterpret_cast<const float4*>(W + (T + r) * LD + col);
      *reinterpret_cast<float4*>(Xg + r * Xld + col) = v;
      if (diag) {
        Di[(col + 0) * T + r] = v.x;
        Di[(col + 1) * T + r] = v.y;
        Di[(col + 2) * T + r] = v.z;
        Di[(col + 3) * T + r] = v.w;
      } else {
        split_store(Xs, Xs + 4096, tc::core_off<64>(r, col), v);
      }
    }
  };
  auto load8 = [](const float* p, float (&v)[8]) {
    const float4 a = *reinterpret_cast<const float4*>(p), b = *reinterpret_cast<const float4*>(p + 4);
    v[0] = a.x;
    v[1] = a.y;
    v[2] = a.z;
    v[3] = a.w;
    v[4] = b.x;
    v[5] = b.y;
    v[6] = b.z;
    v[7] = b.w;
  };
#pragma unroll
  for (int c = 0; c < 8; ++c) x[c] = nx[c] = o[c] = 0.f;
#pragma unroll 1
  for (int b = 0; b < NB; ++b) {
    const int n0 = 8 * b, n1 = n0 + 8;
    const float* last = W + n0 * LD + n0 - 8;   // rows of the diagonal block, columns of the last block
    if (warp == 4) {
      // lane (r, c / 2): entries (r, c), (r, c + 1) of the diagonal block
      float* blk = W + n0 * LD + n0;
      if (b > 0) {
        const int r = lane >> 2, c = 2 * (lane & 3);
        float lr[8], l0[8], l1[8];
        load8(last + r * LD, lr);
        load8(last + c * LD, l0);
        load8(last + (c + 1) * LD, l1);
        float2 v = *reinterpret_cast<float2*>(blk + r * LD + c);
        float s0 = 0.f, s1 = 0.f;
#pragma unroll
        for (int t = 0; t < 8; ++t) {
          s0 = fmaf(lr[t], l0[t], s0);
          s1 = fmaf(lr[t], l1[t], s1);
        }
        *reinterpret_cast<float2*>(blk + r * LD + c) = make_float2(v.x - s0, v.y - s1);
        __syncwarp();
      }
      if (lane == 0) chol8_fast(blk, kt * T + n0, nk, rinv, fail_flags + k, diag ? boosted : nullptr);
    } else if (warp > 4) {
      if (b > 0) store_block(n0 - 8);
    } else if (tid >= n1) {
      // block column b of this row, all terms
      if (b > 0) {
        const float4 a0 = make_float4(o[0], o[1], o[2], o[3]), a1 = make_float4(o[4], o[5], o[6], o[7]);
#pragma unroll
        for (int c = 0; c < 8; ++c) x[c] = nx[c] - dot8(a0, a1, last + c * LD);
      } else {
        load8(my, x);
      }
      // block column b + 1, the terms of blocks 0 .. b - 1
      if (b + 1 < NB) {
        load8(my + n1, nx);
        const float* next = W + n1 * LD;
#pragma unroll 1
        for (int t = 0; t < n0; t += 8) {
          const float4 a0 = *reinterpret_cast<const float4*>(my + t), a1 = *reinterpret_cast<const float4*>(my + t + 4);
#pragma unroll
          for (int c = 0; c < 8; ++c) nx[c] -= dot8(a0, a1, next + c * LD + t);
        }
        if (tid < n1 + 8) {   // a row of the next diagonal block: for the pivot warp
          *reinterpret_cast<float4*>(my + n1) = make_float4(nx[0], nx[1], nx[2], nx[3]);
          *reinterpret_cast<float4*>(my + n1 + 4) = make_float4(nx[4], nx[5], nx[6], nx[7]);
        }
      }
    }
    __syncthreads();
    if (warp < 4 && tid >= n1) {
      float ri[8];
      load8(rinv, ri);
#pragma unroll
      for (int c = 0; c < 8; ++c) o[c] = x[c];
      const float* lb = W + n0 * LD + n0;
      float lc[8][8];
#pragma unroll
      for (int c = 1; c < 8; ++c) {
        const float4 a = *reinterpret_cast<const float4*>(lb + c * LD);
        lc[c][0] = a.x;
        lc[c][1] = a.y;
        lc[c][2] = a.z;
        lc[c][3] = a.w;
        if (c > 4) {
          const float4 e = *reinterpret_cast<const float4*>(lb + c * LD + 4);
          lc[c][4] = e.x;
          lc[c][5] = e.y;
          lc[c][6] = e.z;
        }
      }
#pragma unroll
      for (int t = 0; t < 8; ++t) {
        o[t] *= ri[t];
#pragma unroll
        for (int c = t + 1; c < 8; ++c) o[c] = fmaf(-o[t], lc[c][t], o[c]);
      }
      const float4 a = make_float4(o[0], o[1], o[2], o[3]), e = make_float4(o[4], o[5], o[6], o[7]);
      *reinterpret_cast<float4*>(my + n0) = a;
      *reinterpret_cast<float4*>(my + n0 + 4) = e;
    }
    __syncthreads();
  }
  if (warp > 4) store_block(T - 8);
}

// One launch per tile step: the CTAs of panel kt + 1 first (their chain sets the step's time), then the trailing update
// of step kt; both read column kt, finished by the launch before.  kt = -1: panel 0 alone; FIRST: kt = 0.  The next
// step's CTAs start under programmatic dependent launch: they read their task while this step's last CTAs finish.
// Factorisation stage, before (panel and update launches on two streams, scaled copy, inverses of the diagonal
// tiles) -> now: 12 clusters of 83 cameras 357 -> 207 us, 10 of 100 404 -> 235, 13 uneven of up to 297 2186 -> 924,
// one of 400 1560 -> 702, 67 of 90 1057 -> 680.  Of it: the panel 98 us of 357 (12 clusters), update epilogue and no
// scaled copy 2 (13 uneven: 190 of 2186), one launch per step 28, dependent launch 16, split operands 4 (13 uneven:
// 272).  Panels stacked with the
// tiles below them also where they outnumber the SMs: a separate launch for the diagonal tiles (the split panel)
// would put the update before the tiles below (67 clusters: 819 us split on two streams, 815 one launch).
template <bool FIRST>
__global__ void __launch_bounds__(PTC_THREADS, 2) k_step_tc(float* L, float* Dinv, uint32_t* split,
                                                            const double* __restrict__ S,
                                                            const double* scale, DevProblem P,
                                                            const int2* panels, int npanels, const int2* updates,
                                                            int kt, int* fail_flags, int* boosted, int64_t v_total) {
  extern __shared__ __align__(128) uint32_t step_smem[];
  __shared__ __align__(16) StepShared hs;
  const bool panel = (int)blockIdx.x < npanels;
  const int2 it = panel ? panels[blockIdx.x] : updates[blockIdx.x - npanels];
  const TileTask task{it.x, it.y, P.cluster_np[it.x], P.cluster_n[it.x], P.S_off[it.x], P.v_off[it.x]};
  if (threadIdx.x == 0) {
    tc::mbar_init(&hs.mbar_load, 1);
    tc::mbar_init(&hs.mbar, 1);
  }
  if (threadIdx.x < 32) tc::tmem_alloc(&hs.taddr, STEP_TMEM);
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  // the next step's CTAs may take free SMs and prepare as above; what the launch before wrote, from here on
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
  if (panel)
    panel_tc(step_smem, hs, L, Dinv, split, S, scale, task, kt + 1, fail_flags, boosted, v_total, P.wait_ns);
  else
    update_pair_tc<FIRST>(step_smem, hs, L, split, S, scale, task, kt, fail_flags, v_total, P.wait_ns);
}

// ------------------------------------------------------------------------------------------------------
// Persistent factorisation (FP32 factor, T = 64): one thread-block cluster of FCS CTAs per camera cluster
// runs every tile step of that cluster in one launch.  Tile (i, j) of the lower triangle belongs to CTA
// (i (i + 1) / 2 + j) mod FCS for the whole factorisation (round robin over the tiles, so every step's work
// spreads over the CTAs).  Step kt:
//   1. the owner of (kt, kt) factors the tile (factor_diag_tile; every update of it has been applied by the
//      same CTA) and inverts it (tile_inverse), writing Y = L_kt,kt^-1 and Y^T to Dinv for the solves;
//   2. cluster barrier; every CTA forms its tiles below the diagonal, L_i,kt = A_i,kt Y^T;
//   3. cluster barrier; every CTA applies A_i,j -= L_i,kt L_j,kt^T to its tiles kt < j <= i.
// Between CTAs only the finished column kt (after barrier 2) and Y (after barrier 1) travel, through L2: they
// are read with L1-bypassing loads, after a device-scope fence and the cluster barrier.  Every CTA runs the
// same number of barriers (2 per step).  Replaces the per-step panel / update launches and the separate
// inverses of the diagonal tiles.
constexpr int FCS = 8;

template <int T>
struct ClusterFactorLayout {
  static constexpr int LDA = T + 1;             // diagonal phase: Ad, Y [T][LDA], Z [T * T / 2]
  static constexpr int LD = T + 4;              // product phases: two [T][LD] tiles (16-byte rows)
  static constexpr size_t diag_bytes = sizeof(float) * (2 * (size_t)T * LDA + (size_t)T * T / 2);
  static constexpr size_t prod_bytes = sizeof(float) * 2 * (size_t)T * LD;
  static constexpr size_t bytes = diag_bytes > prod_bytes ? diag_bytes : prod_bytes;
};

__device__ __forceinline__ int factor_tile_owner(int i, int j) { return (i * (i + 1) / 2 + j) % FCS; }

// The 16-byte pieces of a T x T tile that thread t loads (T * T / 4 / 256 of them): piece u is row
// (t + 256 u) % T, columns 4 ((t + 256 u) / T) .. + 3.  Loads first (all in flight at once), stores after.
template <int T>
struct TilePieces {
  static constexpr int N = T * T / 4 / 256;
  float4 v[N];
};
template <int T, bool CG>
__device__ __forceinline__ void tile_pieces_load(TilePieces<T>& t, const float* src, size_t ld) {
#pragma unroll
  for (int u = 0; u < TilePieces<T>::N; ++u) {
    const int q = threadIdx.x + 256 * u, r = q % T, c4 = 4 * (q / T);
    const float4* p = reinterpret_cast<const float4*>(src + (size_t)r * ld + c4);
    t.v[u] = CG ? __ldcg(p) : *p;
  }
}
// dst[c][r] = tile[r][c] (consecutive threads write consecutive r: consecutive banks)
template <int T, int LD>
__device__ __forceinline__ void tile_pieces_store_transposed(float (*dst)[LD], const TilePieces<T>& t) {
#pragma unroll
  for (int u = 0; u < TilePieces<T>::N; ++u) {
    const int q = threadIdx.x + 256 * u, r = q % T, c4 = 4 * (q / T);
    dst[c4][r] = t.v[u].x;
    dst[c4 + 1][r] = t.v[u].y;
    dst[c4 + 2][r] = t.v[u].z;
    dst[c4 + 3][r] = t.v[u].w;
  }
}
// the R x R block (rows tr R + a, columns tc R ..) that the thread updates, as R 16-byte pieces
template <int T>
__device__ __forceinline__ void block_load(float4 (&b)[T / 16], const float* dst, size_t ld) {
  const int tr = threadIdx.x >> 4, tc = threadIdx.x & 15;
#pragma unroll
  for (int a = 0; a < T / 16; ++a) b[a] = *reinterpret_cast<const float4*>(dst + (size_t)(tr * (T / 16) + a) * ld + tc * (T / 16));
}

// acc[a][b] = sum_m X[m][tr R + a] Y[m][tc R + b] over the T rows m of two transposed tiles
template <int T, int LD>
__device__ __forceinline__ void tile_product(const float (*X)[LD], const float (*Y)[LD], float (&acc)[T / 16][T / 16]) {
  constexpr int R = T / 16;
  const int tr = threadIdx.x >> 4, tc = threadIdx.x & 15;
#pragma unroll
  for (int a = 0; a < R; ++a)
#pragma unroll
    for (int b = 0; b < R; ++b) acc[a][b] = 0.f;
#pragma unroll 4
  for (int m = 0; m < T; ++m) {
    float xv[R], yv[R];
    load_vec<float, R>(&X[m][tr * R], xv);
    load_vec<float, R>(&Y[m][tc * R], yv);
#pragma unroll
    for (int a = 0; a < R; ++a)
#pragma unroll
      for (int b = 0; b < R; ++b) acc[a][b] += xv[a] * yv[b];
  }
}

template <int T>
__global__ void __launch_bounds__(256) k_chol_cluster(float* L, float* Dinv, DevProblem P, const int* cluster_items,
                                                      int* fail_flags, int* boosted, int64_t v_total) {
  namespace cg = cooperative_groups;
  using CL = ClusterFactorLayout<T>;
  constexpr int R = T / 16, LDA = CL::LDA, LD = CL::LD;
  cg::cluster_group cluster = cg::this_cluster();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float(*Ad)[LDA] = reinterpret_cast<float(*)[LDA]>(smem_raw);   // diagonal phase
  float(*Y)[LDA] = Ad + T;
  float* Z = reinterpret_cast<float*>(Y + T);
  float(*X1)[LD] = reinterpret_cast<float(*)[LD]>(smem_raw);   // product phases (alias the diagonal phase)
  float(*X2)[LD] = X1 + T;
  __shared__ float rinv2[2][8];
  const int rank = (int)cluster.block_rank();
  const int k = cluster_items[blockIdx.x / FCS];
  const int np = P.cluster_np[k], nk = P.cluster_n[k], nt = np / T;
  float* A = L + P.S_off[k];
  float* Di = Dinv + (size_t)P.v_off[k] * T;
  float* DiT = Di + v_total * T;
  const int tid = threadIdx.x, tr = tid >> 4, tc = tid & 15;
  auto tile = [&](int i, int j) { return A + (size_t)(i * T) * np + j * T; };
  // the diagonal tile kt and its inverse, by its owner (every update of the tile is this CTA's own)
  auto diagonal = [&](int kt) {
    const float* src = tile(kt, kt);
    for (int idx = tid; idx < T * T; idx += 256) {
      const int r = idx / T, c = idx - (idx / T) * T;
      Ad[r][c] = c <= r ? src[(size_t)r * np + c] : 0.f;
      Y[r][c] = 0.f;
    }
    __syncthreads();
    factor_diag_tile<float, T>(Ad, rinv2, kt * T, nk, fail_flags + k, boosted);
    tile_inverse<float, T>(Ad, Y, Z);
    float* d = Di + (size_t)kt * T * T;
    float* dT = DiT + (size_t)kt * T * T;
    for (int idx = tid; idx < T * T; idx += 256) {
      const int r = idx / T, c = idx - (idx / T) * T;
      d[idx] = Y[r][c];
      dT[idx] = Y[c][r];
    }
    __syncthreads();
  };
  if (factor_tile_owner(0, 0) == rank) diagonal(0);
  for (int kt = 0; kt < nt; ++kt) {
    // 1. the diagonal tile kt is factored: at the start (kt = 0) or, one step ahead, by its owner during the
    //    trailing update of step kt - 1 (look-ahead)
    __threadfence();
    cluster.sync();
    // 2. the tiles below the diagonal: L_i,kt = A_i,kt Y^T
    bool have_yt = false;
    for (int i = kt + 1; i < nt; ++i) {
      if (factor_tile_owner(i, kt) != rank) continue;
      TilePieces<T> a_ik, yt;
      tile_pieces_load<T, false>(a_ik, tile(i, kt), np);   // this CTA's own tile
      if (!have_yt) tile_pieces_load<T, true>(yt, DiT + (size_t)kt * T * T, T);   // Y^T, row-major in DiT
      tile_pieces_store_transposed<T, LD>(X1, a_ik);
      if (!have_yt) {   // X2[m][c] = (Y^T)[m][c]: the pieces go in untransposed
#pragma unroll
        for (int u = 0; u < TilePieces<T>::N; ++u) {
          const int q = tid + 256 * u, r = q % T, c4 = 4 * (q / T);
          *reinterpret_cast<float4*>(&X2[r][c4]) = yt.v[u];
        }
        have_yt = true;
      }
      __syncthreads();
      float acc[R][R];
      tile_product<T, LD>(X1, X2, acc);
      float* dst = tile(i, kt);
#pragma unroll
      for (int a = 0; a < R; ++a)
        *reinterpret_cast<float4*>(dst + (size_t)(tr * R + a) * np + tc * R) =
            make_float4(acc[a][0], acc[a][1], acc[a][2], acc[a][3]);
      __syncthreads();   // X1 is reloaded next
    }
    __threadfence();
    cluster.sync();
    // 3. trailing update of this CTA's tiles kt < j <= i; the owner of the next diagonal tile updates it first
    //    and factors it before its other tiles (look-ahead)
    if (kt + 1 < nt && factor_tile_owner(kt + 1, kt + 1) == rank) {
      TilePieces<T> l1;
      float4 old[R];
      float* dst = tile(kt + 1, kt + 1);
      tile_pieces_load<T, true>(l1, tile(kt + 1, kt), np);
      block_load<T>(old, dst, np);
      tile_pieces_store_transposed<T, LD>(X1, l1);
      __syncthreads();
      float acc[R][R];
      tile_product<T, LD>(X1, X1, acc);
#pragma unroll
      for (int a = 0; a < R; ++a)
        *reinterpret_cast<float4*>(dst + (size_t)(tr * R + a) * np + tc * R) =
            make_float4(old[a].x - acc[a][0], old[a].y - acc[a][1], old[a].z - acc[a][2], old[a].w - acc[a][3]);
      __syncthreads();
      diagonal(kt + 1);
    }
    for (int i = kt + 1; i < nt; ++i) {
      bool have_li = false;
      for (int j = kt + 1; j <= i; ++j) {
        if (factor_tile_owner(i, j) != rank || (i == kt + 1 && j == kt + 1)) continue;
        TilePieces<T> li, lj;
        float4 old[R];
        float* dst = tile(i, j);
        if (!have_li) tile_pieces_load<T, true>(li, tile(i, kt), np);
        tile_pieces_load<T, true>(lj, tile(j, kt), np);
        block_load<T>(old, dst, np);
        if (!have_li) {
          tile_pieces_store_transposed<T, LD>(X1, li);
          have_li = true;
        }
        tile_pieces_store_transposed<T, LD>(X2, lj);
        __syncthreads();
        float acc[R][R];
        tile_product<T, LD>(X1, X2, acc);
#pragma unroll
        for (int a = 0; a < R; ++a)
          *reinterpret_cast<float4*>(dst + (size_t)(tr * R + a) * np + tc * R) =
              make_float4(old[a].x - acc[a][0], old[a].y - acc[a][1], old[a].z - acc[a][2], old[a].w - acc[a][3]);
        __syncthreads();   // X2 (and X1 at the next i) are reloaded
      }
    }
  }
}

// ------------------------------------------------------------------------------------------------------
template <typename F>
__device__ F warp_sum(F v) {
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) v += __shfl_xor_sync(FULL_MASK, v, d);
  return v;
}

// x := D^-1/2 (L L^T)^-1 D^-1/2 rhs  (accumulate = 0) or x += ... (accumulate = 1).
// One thread-block cluster of CS CTAs per camera cluster.  Each CTA keeps the whole vector in shared
// memory; at tile step `it` CTA `rank` forms the partial product of the tiles it owns (tile columns j <
// it with j = rank mod CS for the forward pass, tile rows j > it for the backward pass), the partials are
// exchanged through distributed shared memory after one cluster barrier, and every CTA applies the stored
// inverse of the diagonal tile redundantly, so the next step needs no further synchronisation.  The tiles
// do not depend on the vector: the owned tiles of the next steps (up to SOLVE_PF of them each) and their
// diagonal inverses are copied into shared memory (cp.async) while step it computes, `nst` stages deep:
// three (two steps ahead) when the launch is one wave of CTAs, two otherwise, where the smaller shared
// memory lets two CTAs share an SM and the waves halve.
constexpr int SOLVE_PF = 2;

template <typename F, int T>
struct SolveLayout {
  static constexpr int LDT = T + 16 / (int)sizeof(F);   // padded rows, 16-byte aligned
  static constexpr size_t tile_elems = (size_t)T * LDT;
  // per stage [SOLVE_PF tiles + 1 diagonal inverse][T][LDT]; the stages are followed by the vector y
  static constexpr size_t stage_bytes = sizeof(F) * (SOLVE_PF + 1) * tile_elems;
};

__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait1() { asm volatile("cp.async.wait_group 1;\n" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait2() { asm volatile("cp.async.wait_group 2;\n" ::: "memory"); }

// T x T tile at src (row stride ld elements) into padded shared rows
template <typename F, int T>
__device__ __forceinline__ void prefetch_tile(F* dst, const F* src, size_t ld) {
  constexpr int CH = T * (int)sizeof(F) / 16;   // 16-byte chunks per row
  constexpr int LDT = SolveLayout<F, T>::LDT;
  for (int q = threadIdx.x; q < T * CH; q += blockDim.x) {
    const int r = q / CH, c = q - (q / CH) * CH;
    cp_async16(dst + (size_t)r * LDT + c * (16 / sizeof(F)), src + (size_t)r * ld + c * (16 / sizeof(F)));
  }
}

// out[r] = sum_c M[r][c] v[c], M a padded shared tile; 256 / T threads per row
template <typename F, int T>
__device__ __forceinline__ void smem_matvec(const F* M, const F* v, F* out) {
  constexpr int PARTS = 256 / T, LEN = T / PARTS, LDT = SolveLayout<F, T>::LDT;
  const int r = threadIdx.x / PARTS, part = threadIdx.x - (threadIdx.x / PARTS) * PARTS;
  const F* row = M + (size_t)r * LDT + part * LEN;
  F s = F(0);
#pragma unroll
  for (int c = 0; c < LEN; ++c) s += row[c] * v[part * LEN + c];
#pragma unroll
  for (int d = PARTS / 2; d > 0; d >>= 1) s += __shfl_xor_sync(0xffffffffu, s, d);
  if (part == 0) out[r] = s;
}

template <typename F, int T, typename Rreal, int CS>
__global__ void __launch_bounds__(256) k_tri_solve(DevProblem P, const F* L, const F* Dinv, const double* scale,
                                                   const Rreal* rhs, double* x, int accumulate, int64_t v_total,
                                                   int nst) {
  namespace cg = cooperative_groups;
  using SL = SolveLayout<F, T>;
  constexpr int PARTS = 256 / T, LEN = T / PARTS, LDT = SL::LDT;
  cg::cluster_group cluster = cg::this_cluster();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  F* buf = reinterpret_cast<F*>(smem_raw);                   // [nst][SOLVE_PF + 1][T][LDT]
  F* y = buf + nst * (SOLVE_PF + 1) * SL::tile_elems;
  __shared__ F partial[2][T];
  __shared__ F t[T];
  __shared__ F pcol[PARTS][T];
  const int rank = (int)cluster.block_rank();
  const int k = blockIdx.x / CS;
  if (P.sharded && !P.cluster_owned[k]) return;   // the whole thread-block cluster leaves, before any barrier
  const int np = P.cluster_np[k];
  const F* A = L + P.S_off[k];
  const F* Di = Dinv + (size_t)P.v_off[k] * T;
  const F* DiT = Di + v_total * T;
  const double* sk = scale + P.v_off[k];
  const Rreal* rk = rhs + P.v_off[k];
  double* xk = x + P.v_off[k];
  const int nt = np / T;
  const int tid = threadIdx.x;
  auto tile_buf = [&](int stage, int slot) { return buf + ((size_t)stage * (SOLVE_PF + 1) + slot) * SL::tile_elems; };
  // step s = 0 .. 2 nt - 1: forward steps it = s, backward steps it = 2 nt - 1 - s
  auto issue = [&](int s) {
    if (s < 2 * nt) {
      const bool fwd = s < nt;
      const int it = fwd ? s : 2 * nt - 1 - s;
      int m = 0;
      if (fwd) {
        for (int j = rank; j < it && m < SOLVE_PF; j += CS, ++m)
          prefetch_tile<F, T>(tile_buf(s % nst, m), A + (size_t)(it * T) * np + j * T, np);
      } else {
        for (int j = it + 1 + rank; j < nt && m < SOLVE_PF; j += CS, ++m)
          prefetch_tile<F, T>(tile_buf(s % nst, m), A + (size_t)(j * T) * np + it * T, np);
      }
      prefetch_tile<F, T>(tile_buf(s % nst, SOLVE_PF), (fwd ? Di : DiT) + (size_t)it * T * T, T);
    }
    cp_async_commit();
  };
  issue(0);
  if (nst == 3) issue(1);
  for (int i = tid; i < np; i += blockDim.x) y[i] = (F)((double)rk[i] * sk[i]);
  for (int s = 0; s < 2 * nt; ++s) {
    issue(s + nst - 1);   // into the stage step s - 1 used; every thread passed its last barrier
    if (nst == 3)
      cp_async_wait2();
    else
      cp_async_wait1();
    __syncthreads();
    const int st = s % nst;
    const bool fwd = s < nt;
    const int it = fwd ? s : 2 * nt - 1 - s;
    const int r0 = it * T;
    if (fwd) {
      // partial[r] = sum over owned tiles j of L[it][j] y_j: thread (row, part)
      const int r = tid / PARTS, part = tid - (tid / PARTS) * PARTS;
      F acc = F(0);
      int m = 0;
      for (int j = rank; j < it; j += CS, ++m) {
        const F* yj = y + j * T + part * LEN;
        if (m < SOLVE_PF) {
          const F* row = tile_buf(st, m) + (size_t)r * LDT + part * LEN;
#pragma unroll
          for (int c = 0; c < LEN; ++c) acc += row[c] * yj[c];
        } else {
          const F* row = A + (size_t)(r0 + r) * np + j * T + part * LEN;
#pragma unroll
          for (int c = 0; c < LEN; ++c) acc += __ldg(row + c) * yj[c];
        }
      }
#pragma unroll
      for (int d = PARTS / 2; d > 0; d >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, d);
      if (part == 0) partial[s & 1][r] = acc;
    } else {
      // partial[c] = sum over owned tiles j of L[j][it]^T z_j: thread (column, part of the rows)
      const int c = tid % T, part = tid / T;
      F acc = F(0);
      int m = 0;
      for (int j = it + 1 + rank; j < nt; j += CS, ++m) {
        const F* zj = y + j * T + part * LEN;
        if (m < SOLVE_PF) {
          const F* col = tile_buf(st, m) + (size_t)(part * LEN) * LDT + c;
#pragma unroll
          for (int rr = 0; rr < LEN; ++rr) acc += col[(size_t)rr * LDT] * zj[rr];
        } else {
          const F* col = A + (size_t)(j * T + part * LEN) * np + r0 + c;
#pragma unroll
          for (int rr = 0; rr < LEN; ++rr) acc += __ldg(col + (size_t)rr * np) * zj[rr];
        }
      }
      pcol[part][c] = acc;
      __syncthreads();
      if (tid < T) {
        F v = F(0);
#pragma unroll
        for (int q = 0; q < PARTS; ++q) v += pcol[q][tid];
        partial[s & 1][tid] = v;
      }
    }
    cluster.sync();
    for (int r = tid; r < T; r += blockDim.x) {
      F sum = F(0);
#pragma unroll
      for (int q = 0; q < CS; ++q) sum += cluster.map_shared_rank(&partial[s & 1][0], q)[r];
      t[r] = y[r0 + r] - sum;
    }
    __syncthreads();
    // y_it = D_it^-1 t (forward) or D_it^-T t (backward, through the stored transpose)
    smem_matvec<F, T>(tile_buf(st, SOLVE_PF), t, y + r0);
    __syncthreads();
  }
  if (rank == 0)
    for (int i = tid; i < np; i += blockDim.x) {
      const double v = (double)y[i] * sk[i];
      xk[i] = accumulate ? xk[i] + v : v;
    }
  cluster.sync();   // keep this CTA's shared memory alive until every peer has read it
}

// ------------------------------------------------------------------------------------------------------
// The same solve as a data flow (clusters whose accumulators fit in shared memory: up to 94, 168 and 280 tile rows of
// either factor with 2, 4 and 8 CTAs; k_tri_solve beyond): tile row i belongs to CTA i mod CS of the cluster's CS CTAs.
// Forward, the owner of row k finishes t_k = r_k - sum_j L_kj y_j, forms y_k = D_k^-1 t_k and sends it to every CTA with
// a row below k, with asynchronous stores counted by that CTA's mbarrier of step k; whoever has y_k subtracts
// L_ik y_k from its rows i > k, row k + 1 first, whose owner then goes on to y_k+1 before its other rows.  The
// backward pass is the same on reversed indices with L_ki^T and D_k^-T.  A step's chain is two 64 x 64 products by
// 256 threads and one remote store: 0.8 us (12 clusters of 83 cameras) to 1.4 us (one of 400, whose later steps also
// have 7 rows per CTA to update), against 2.4 us with a cluster barrier, a gather of the partial products from all
// CTAs and five block barriers per step.
// Only the mbarrier that it counts on tells that an asynchronous store has arrived (a cluster barrier orders its
// issue).  A piece goes to no CTA that does not wait for it, so
//   - no CTA leaves while a store to it is under way;
//   - x_k never meets y_k on its way to the same place in a CTA: a CTA that gets y_k owns a row i > k, sends x_i only
//     after its forward pass, in which it has waited for y_k, and x_k is formed from x_i.
// Nothing depends on a tile's address on the vector, so each thread keeps its elements of the next NB tiles in registers (loads in flight while it waits for y_k).
// NB = 4 tiles of the FP32 factor (64 registers; 3 and 4 alike at 15 tile rows, 4 better beyond, 5 spills).
// Solve stage with one refinement step, before (k_tri_solve, one residual CTA per tile row) -> now: 12 clusters of 83
// cameras 180 -> 66 us, 13 uneven of up to 297 753 -> 285, one of 400 1053 -> 310, 67 of 90 350 -> 197; FP64, 4 clusters
// of 75 387 -> 201.  With every piece sent to all CTAs, and each waiting for all of a pass before the next and before it
// leaves: 69, 295, 324 and 202.
template <typename F, int T> struct PushLayout {
  static constexpr int V = 16 / (int)sizeof(F);          // elements per 16-byte load
  static constexpr int PARTS = 256 / T;                  // row products: threads per row
  static constexpr int NL = T * T / 256 / V;             // 16-byte loads of a tile per thread
  static constexpr int CG = T / V, RPN = 256 / CG;       // column products: column groups, row parts of NL rows
  static constexpr int NB = NL == 1 ? 6 : 4;             // tiles in registers or in flight per thread
  static size_t bytes(int nt, int cs) {
    const int slots = (nt + cs - 1) / cs;
    return 16 * (size_t)nt + sizeof(F) * ((size_t)nt * T + (size_t)slots * (T + 256 * V) + 9 * (size_t)T) + 16;
  }
};

template <typename F, int N>
__device__ __forceinline__ void load16s(const F* p, F* v) {   // one 16-byte load (N = 4 floats or 2 doubles)
  if constexpr (sizeof(F) == 4) {
    const float4 t = *reinterpret_cast<const float4*>(p);
    v[0] = t.x;
    v[1] = t.y;
    v[2] = t.z;
    v[3] = t.w;
  } else {
    const double2 t = *reinterpret_cast<const double2*>(p);
    v[0] = t.x;
    v[1] = t.y;
  }
}

template <typename F, int T, typename Rreal, int CS>
__global__ void __launch_bounds__(256, T == 64 ? 2 : 3) k_tri_push(DevProblem P, const F* L, const F* Dinv,
                                                     const double* scale, const Rreal* rhs,
                                                     double* x, double* rcopy, int accumulate, int64_t v_total,
                                                     int max_nt, int* fail_flags) {
  namespace cg = cooperative_groups;
  using PL = PushLayout<F, T>;
  constexpr int V = PL::V, PARTS = PL::PARTS, NL = PL::NL, CG = PL::CG, NB = PL::NB;
  chain_begin();
  cg::cluster_group cluster = cg::this_cluster();
  const int rank = (int)cluster.block_rank();
  const int k = blockIdx.x / CS;
  if (P.sharded && !P.cluster_owned[k]) return;   // the whole thread-block cluster leaves, before any barrier
  const int np = P.cluster_np[k], nt = np / T;
  const F* A = L + P.S_off[k];
  const F* Di = Dinv + (size_t)P.v_off[k] * T;
  const F* DiT = Di + v_total * T;
  const double* sk = scale + P.v_off[k];
  const Rreal* rk = rhs + P.v_off[k];
  double* xk = x + P.v_off[k];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int slots = (max_nt + CS - 1) / CS;
  uint64_t* mbar = reinterpret_cast<uint64_t*>(smem_raw);        // [2][max_nt]: y_k, then x_k, has arrived
  F* vec = reinterpret_cast<F*>(smem_raw + 16 * (size_t)max_nt);   // [max_nt][T] y, overwritten by x
  F* own = vec + (size_t)max_nt * T;                               // [slots][T] r, then y, of this CTA's rows
  F* acc = own + (size_t)slots * T;                                // [slots][256][V] per-thread sums of products
  F* red = acc + (size_t)slots * 256 * V;                          // [8][T]
  F* tv = red + 8 * T;                                             // [T]
  for (int i = tid; i < 2 * nt; i += 256) {
    const int b = i < nt ? i : max_nt + i - nt;
    tc::mbar_init(mbar + b, 1);
    tc::mbar_arrive_expect(mbar + b, (uint32_t)(T * sizeof(F)));
  }
  const int nown = rank < nt ? (nt - 1 - rank) / CS + 1 : 0;
  for (int e = tid; e < nown * T; e += 256) {
    const int g = (rank + CS * (e / T)) * T + e % T;
    own[e] = (F)((double)rk[g] * sk[g]);
    if (rcopy) rcopy[P.v_off[k] + g] = (double)rk[g];
  }
  for (int e = tid; e < nown * 256 * V; e += 256) acc[e] = F(0);
  __syncthreads();
  cluster.sync();   // every CTA's barriers are set up before the first remote store
  const int row = tid / PARTS, part = tid - row * PARTS;   // row products
  const int cgp = tid % CG, rp = tid / CG;                 // column products: rows rp NL ..
  bool dead = false;
  constexpr int PEERS = (CS + PARTS - 1) / PARTS;
  uint32_t rvec[PEERS], rbar[PEERS];   // the peers this thread sends to
#pragma unroll
  for (int u = 0; u < PEERS; ++u) {
    const uint32_t peer = (uint32_t)min(part + PARTS * u, CS - 1);
    rvec[u] = tc::map_rank(tc::smem_u32(vec), peer);
    rbar[u] = tc::map_rank(tc::smem_u32(mbar), peer);
  }
  // Indices i of a pass run upwards: the tile row i (forward) or nt - 1 - i (backward).  The largest of CTA r's, which
  // are equal mod CS; it takes the pieces of the indices before it (-1: it has no row).
  auto last_of = [&](int r, bool fwd) {
    const int first = fwd ? r : ((nt - 1 - r) % CS + CS) % CS;
    return r < CS && r < nt ? first + CS * ((nt - 1 - first) / CS) : -1;
  };
  // one pass
  auto pass = [&](auto fwd_c) {
    constexpr bool FWD = decltype(fwd_c)::value;
    const int me = FWD ? rank : ((nt - 1 - rank) % CS + CS) % CS;   // this CTA's pass indices are me mod CS
    if (nown == 0) return;
    const int last = last_of(rank, FWD);
    int rlast[PEERS];
#pragma unroll
    for (int u = 0; u < PEERS; ++u) rlast[u] = last_of(part + PARTS * u, FWD);
    // tasks: update of index i by the vector piece of index kk (i > kk), or the diagonal product of index i (diag)
    struct Task {
      int i, kk;
      bool diag, end;
    };
    auto first_of = [&](int kk) {   // the first task of step kk
      Task t{0, kk, false, kk >= last};
      const int d = ((me - (kk + 1)) % CS + CS) % CS;
      t.i = kk + 1 + d;
      return t;
    };
    auto next = [&](const Task& t) {
      if (t.end) return t;
      if (!t.diag && t.i == t.kk + 1) return Task{t.i, t.kk, true, false};
      if (t.diag && t.kk < 0) return first_of(0);
      return t.i + CS < nt ? Task{t.i + CS, t.kk, false, false} : first_of(t.kk + 1);
    };
    auto at = [&](int i) { return FWD ? i : nt - 1 - i; };
    auto fetch = [&](const Task& t, F (&b)[NL * V]) {
      if (t.end) return;
      if (t.diag || FWD) {
        const F* src = t.diag ? (FWD ? Di : DiT) + (size_t)at(t.i) * T * T + (size_t)row * T
                              : A + (size_t)(at(t.i) * T + row) * np + at(t.kk) * T;
#pragma unroll
        for (int u = 0; u < NL; ++u) load16s<F, V>(src + V * (part + PARTS * u), b + V * u);
      } else {
        const F* src = A + (size_t)(at(t.kk) * T + rp * NL) * np + at(t.i) * T + V * cgp;
#pragma unroll
        for (int u = 0; u < NL; ++u) load16s<F, V>(src + (size_t)u * np, b + V * u);
      }
    };
    auto row_dot = [&](const F (&cur)[NL * V], const F* v) {   // this thread's part of its row's product with v
      F s = F(0);
#pragma unroll
      for (int u = 0; u < NL; ++u)
#pragma unroll
        for (int e = 0; e < V; ++e) s += cur[V * u + e] * v[V * (part + PARTS * u) + e];
      return s;
    };
    auto row_sum = [&](F s) {   // over the threads of a row
#pragma unroll
      for (int d = PARTS / 2; d > 0; d >>= 1) s += __shfl_xor_sync(FULL_MASK, s, d);
      return s;
    };
    // the tiles of the next NB tasks, in flight or in registers; buffer b serves tasks b, b + NB, ..
    F buf[NB][NL * V];
    Task tk[NB];
    tk[0] = me == 0 ? Task{0, -1, true, false} : first_of(0);
#pragma unroll
    for (int b = 0; b < NB; ++b) {
      if (b > 0) tk[b] = next(tk[b - 1]);
#pragma unroll
      for (int u = 0; u < NL * V; ++u) buf[b][u] = F(0);
      fetch(tk[b], buf[b]);
    }
    Task tn = next(tk[NB - 1]);
    int have = -1;   // the last step whose piece has arrived
    auto work = [&](const Task& t0, const F (&cur)[NL * V]) {
      const int slot = (at(t0.i) - rank) / CS;
      if (t0.diag) {
        F t;
        if constexpr (FWD) {
          t = own[slot * T + row] - row_sum(acc[(slot * 256 + tid) * V]);
          if (part == 0) tv[row] = t;
        } else {
          F a[V];
#pragma unroll
          for (int e = 0; e < V; ++e) a[e] = acc[(slot * 256 + tid) * V + e];
#pragma unroll
          for (int d = CG; d < 32; d <<= 1)
#pragma unroll
            for (int e = 0; e < V; ++e) a[e] += __shfl_xor_sync(FULL_MASK, a[e], d);
          if (lane < CG) {
#pragma unroll
            for (int e = 0; e < V; ++e) red[warp * T + V * cgp + e] = a[e];
          }
          __syncthreads();
          if (tid < T) {
            F s = F(0);
#pragma unroll
            for (int w = 0; w < 8; ++w) s += red[w * T + tid];
            tv[tid] = own[slot * T + tid] - s;
          }
        }
        __syncthreads();
        const F y = row_sum(row_dot(cur, tv));
        const int g = at(t0.i) * T + row;
#pragma unroll
        for (int u = 0; u < PEERS; ++u)
          if (rlast[u] > t0.i)
            tc::st_async(rvec[u] + (uint32_t)(g * sizeof(F)), y, rbar[u] + (uint32_t)(8 * ((FWD ? 0 : max_nt) + at(t0.i))));
        if (part == 0) {
          if constexpr (FWD) {
            own[slot * T + row] = y;
          } else {
            const double v = (double)y * sk[g];
            xk[g] = accumulate ? xk[g] + v : v;
          }
        }
      } else {
        if (t0.kk > have) {
          if (!dead) dead = !tc::mbar_wait_bounded(mbar + (FWD ? 0 : max_nt) + at(t0.kk), 0, P.wait_ns);
          have = t0.kk;
        }
        const F* v = vec + (size_t)at(t0.kk) * T;
        F* a = acc + (size_t)(slot * 256 + tid) * V;
        if constexpr (FWD) {
          a[0] += row_dot(cur, v);
        } else {
          F s[V];
#pragma unroll
          for (int e = 0; e < V; ++e) s[e] = a[e];
#pragma unroll
          for (int u = 0; u < NL; ++u) {
            const F xv = v[rp * NL + u];
#pragma unroll
            for (int e = 0; e < V; ++e) s[e] += cur[V * u + e] * xv;
          }
#pragma unroll
          for (int e = 0; e < V; ++e) a[e] = s[e];
        }
      }
    };
    for (bool more = true; more;) {
#pragma unroll
      for (int b = 0; b < NB; ++b) {
        if (tk[b].end) {
          more = false;
          break;
        }
        work(tk[b], buf[b]);
        tk[b] = tn;
        fetch(tn, buf[b]);
        tn = next(tn);
      }
    }
  };
  pass(std::true_type{});
  __syncthreads();   // y of this CTA's rows, before the backward pass reads it
  for (int e = tid; e < nown * 256 * V; e += 256) acc[e] = F(0);   // thread-private up to the reductions, but indexed by
  __syncthreads();                                                 // another layout here
  pass(std::false_type{});
  if (dead) {   // a wait gave up: the step is rejected.  What is on its way to this CTA still has to arrive
    atomicOr(fail_flags + k, FAIL_WAIT);
    for (int i = 0; i < last_of(rank, true); ++i) tc::mbar_wait_bounded(mbar + i, 0, tc::WAIT_NS);
    for (int i = 0; i < last_of(rank, false); ++i) tc::mbar_wait_bounded(mbar + max_nt + nt - 1 - i, 0, tc::WAIT_NS);
  }
  cluster.sync();
}

// Device figures, read by configure_solve_kernels.
static int g_num_sms = 0, g_smem_optin = 0;

// Shared memory of one solve CTA: nst stages, the vector, and the static arrays (partial[2][T], t[T],
// pcol[256 / T][T]).
template <typename F, int T>
size_t solve_cta_bytes(int nst, int max_np) {
  return nst * SolveLayout<F, T>::stage_bytes +
         sizeof(F) * ((size_t)max_np + (3 + 256 / T) * (size_t)T);
}

template <typename F, int T>
int solve_stages(int l, int max_np, int cs) {
  const bool one_wave = (int64_t)l * cs <= g_num_sms;
  return one_wave && solve_cta_bytes<F, T>(3, max_np) <= (size_t)g_smem_optin ? 3 : 2;
}

// r = rhs copied to rcopy (unless null) along the way
template <typename F, int T, typename Rreal>
void launch_tri_solve(const DevProblem& P, const F* L, const F* Dinv, const double* scale, const Rreal* rhs,
                      double* x, double* rcopy, int accumulate, int max_np, int64_t v_total, int cs, int* fail_flags,
                      bool after_kernel, cudaStream_t stream) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(P.l * cs);
  cfg.blockDim = dim3(256);
  cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = cs;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  const int max_nt = max_np / T;
  const size_t push = PushLayout<F, T>::bytes(max_nt, cs);
  if (push <= (size_t)g_smem_optin) {
    cfg.dynamicSmemBytes = push;
    cfg.numAttrs = after_kernel && chained(P) ? 2 : 1;
    auto* kern = cs == 2 ? k_tri_push<F, T, Rreal, 2> : cs == 4 ? k_tri_push<F, T, Rreal, 4> : k_tri_push<F, T, Rreal, 8>;
    cudaLaunchKernelEx(&cfg, kern, P, L, Dinv, scale, rhs, x, rcopy, accumulate, v_total, max_nt, fail_flags);
    return;
  }
  // clusters too large for the accumulators
  if (rcopy) cudaMemcpyAsync(rcopy, rhs, (size_t)v_total * sizeof(double), cudaMemcpyDeviceToDevice, stream);
  const int nst = solve_stages<F, T>(P.l, max_np, cs);
  cfg.dynamicSmemBytes = nst * SolveLayout<F, T>::stage_bytes + sizeof(F) * (size_t)max_np;
  auto* kern = cs == 2 ? k_tri_solve<F, T, Rreal, 2> : cs == 4 ? k_tri_solve<F, T, Rreal, 4> : k_tri_solve<F, T, Rreal, 8>;
  cudaLaunchKernelEx(&cfg, kern, P, L, Dinv, scale, rhs, x, accumulate, v_total, nst);
}

// r = b - S x (FP64) with S symmetric, lower triangle stored; r was set to b before.  One CTA per
// (cluster, 32-row tile row I, RES_TILES of its tiles); its 4 warps take the tiles (I, J), J <= I, in turn.  A warp
// stages the 32 x 32 tile in shared memory with coalesced row loads, then lane l forms both the row sum of tile row l
// (S_IJ x_J, kept in registers over the warp's tiles) and the column sum of tile column l (S_IJ^T x_I,
// added atomically to r_J; on the diagonal tile only below the diagonal).
constexpr int RES_WARPS = 4;

template <typename Sreal>
__global__ void __launch_bounds__(32 * RES_WARPS) k_residual(DevProblem P, const Sreal* S, const double* x,
                                                             double* r, const int2* items) {
  __shared__ double T[RES_WARPS][32][33];
  __shared__ double xs[RES_WARPS][32];
  __shared__ double xi[32];
  __shared__ double red[RES_WARPS][32];
  chain_begin();
  const int2 it = items[blockIdx.x];
  const int k = it.x, I = it.y & 0xffff, J0 = RES_TILES * (it.y >> 16);
  const int np = P.cluster_np[k], nk = P.cluster_n[k];
  const Sreal* Sk = S + P.S_off[k];
  const double* xk = x + P.v_off[k];
  double* rk = r + P.v_off[k];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int i0 = 32 * I;
  if (warp == 0) xi[lane] = (i0 + lane < nk) ? xk[i0 + lane] : 0.0;
  __syncthreads();
  double rowacc = 0.0;
  const int J1 = min(I, J0 + RES_TILES - 1);
  for (int J = J0 + warp; J <= J1; J += RES_WARPS) {
    const int j0 = 32 * J;
    const int col = j0 + lane;
    for (int rr = 0; rr < 32; ++rr) {
      const int row = i0 + rr;
      T[warp][rr][lane] = (row < nk && col < nk && col <= row) ? (double)Sk[(size_t)row * np + col] : 0.0;
    }
    xs[warp][lane] = (col < nk) ? xk[col] : 0.0;
    __syncwarp();
    double rs = 0.0, cs = 0.0;
#pragma unroll 8
    for (int c = 0; c < 32; ++c) rs += T[warp][lane][c] * xs[warp][c];
    if (J < I) {
#pragma unroll 8
      for (int rr = 0; rr < 32; ++rr) cs += T[warp][rr][lane] * xi[rr];
    } else {
      for (int rr = lane + 1; rr < 32; ++rr) cs += T[warp][rr][lane] * xi[rr];
    }
    rowacc += rs;
    if (col < nk && cs != 0.0) atomicAdd(rk + col, -cs);
    __syncwarp();
  }
  red[warp][lane] = rowacc;
  __syncthreads();
  if (warp == 0) {
    double t = 0.0;
#pragma unroll
    for (int w = 0; w < RES_WARPS; ++w) t += red[w][lane];
    if (i0 + lane < nk) atomicAdd(rk + i0 + lane, -t);
  }
}

// ------------------------------------------------------------------------------------------------------
// Host launchers

// A launch of `threads` threads (256 for launch_prio) with a scheduling priority (kept by graph capture as a
// node attribute): the panels on the critical path go first, the trailing updates fill the remaining SMs.
template <typename... KArgs, typename... Args>
void launch_prio_n(void (*kernel)(KArgs...), int grid, int threads, size_t smem, cudaStream_t stream, int prio,
                   Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributePriority;
  attr[0].val.priority = prio;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}

template <typename... KArgs, typename... Args>
void launch_prio(void (*kernel)(KArgs...), int grid, size_t smem, cudaStream_t stream, int prio, Args... args) {
  launch_prio_n(kernel, grid, 256, smem, stream, prio, args...);
}
// A panel CTA is bound by the latency of its column chain: a second panel CTA on the same SM would halve
// the speed of both.  When a tile step's panels fit on the SMs one each, their dynamic shared memory is
// raised above half of an SM's so that they do take one SM each; a step with more panels than SMs keeps
// the plain size, so that the SMs hold several and the waves stay few (figures set by
// configure_solve_kernels).
static size_t g_panel_min_smem = 0;

template <typename F, int T>
size_t panel_smem(int npn = 0) {
  return npn <= g_num_sms ? std::max(PanelLayout<F, T>::bytes, g_panel_min_smem) : PanelLayout<F, T>::bytes;
}

// whether the factorisation runs as tensor-core steps (k_step_tc)
template <typename F, int T>
bool tensor_steps(const CholPlan& plan) {
  return sizeof(F) == 4 && T == 64 && plan.update_tc && !plan.persistent;
}

template <typename F, int T>
void launch_factor_t(const DevProblem& P, const double* S, const FactorBuffers& fb, const CholPlan& plan,
                     cudaStream_t stream) {
  using Sreal = double;
  F* L = reinterpret_cast<F*>(fb.L);
  F* Dinv = reinterpret_cast<F*>(fb.Dinv);
  dim3 g1(std::max(1, std::min(plan.max_np / 256 + 1, 64)), P.l);
  k_diag_scale<Sreal><<<g1, 256, 0, stream>>>(P, S, fb.scale);
  dim3 g2(std::min(plan.max_np, 1024), P.l);
  const bool tcf = tensor_steps<F, T>(plan);   // they read S' themselves, no scaled copy
  // the first tile column now (the first panels read it); with more tile steps, the rest of the copy runs
  // on the side stream beside panel 0, and panel 1 waits for it
  bool copy_beside = !tcf && plan.nsteps > 1 && plan.ev_copy != nullptr;
  if constexpr (sizeof(F) == 4 && T == 64) copy_beside = copy_beside && !plan.persistent;
  if (!tcf) k_scaled_copy<Sreal, F><<<g2, 256, 0, stream>>>(P, S, fb.scale, L, 0, copy_beside ? T : INT_MAX);
  // panels on `stream`; the trailing updates (all tiles but the next column, which the next panel updates
  // itself) on the side stream, so that update kt overlaps panel kt + 1.  Panel kt + 2 waits for update kt.
  if constexpr (sizeof(F) == 4 && T == 64) {
    if (plan.persistent) {   // every tile step of every cluster in one launch of 8-CTA thread-block clusters
      if (plan.n_cluster_items > 0) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(plan.n_cluster_items * FCS);
        cfg.blockDim = dim3(256);
        cfg.dynamicSmemBytes = ClusterFactorLayout<T>::bytes;
        cfg.stream = stream;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = FCS;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        cudaLaunchKernelEx(&cfg, k_chol_cluster<T>, reinterpret_cast<float*>(L), reinterpret_cast<float*>(Dinv), P,
                           plan.cluster_items, fb.fail_flags, fb.boosted, fb.v_total);
      }
      return;
    }
  }
  if constexpr (sizeof(F) == 4 && T == 64) {
    if (tcf) {
      constexpr size_t smem = std::max(PTC_SMEM, TCU_SMEM);
      for (int kt = -1; kt + 1 < plan.nsteps; ++kt) {
        const int npn = plan.h_panel_off[kt + 2] - plan.h_panel_off[kt + 1];
        const int nu = kt < 0 ? 0 : plan.h_update_off[kt + 1] - plan.h_update_off[kt];
        if (npn + nu == 0) continue;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(npn + nu);
        cfg.blockDim = dim3(PTC_THREADS);
        cfg.dynamicSmemBytes = smem;
        cfg.stream = stream;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[0].val.programmaticStreamSerializationAllowed = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        cudaLaunchKernelEx(&cfg, kt == 0 ? k_step_tc<true> : k_step_tc<false>, reinterpret_cast<float*>(L),
                           reinterpret_cast<float*>(Dinv), fb.split, S, (const double*)fb.scale, P,
                           plan.panel_items + plan.h_panel_off[kt + 1], npn,
                           plan.update_items + (kt < 0 ? 0 : plan.h_update_off[kt]), kt, fb.fail_flags, fb.boosted,
                           fb.v_total);
      }
      return;
    }
  }
  cudaStream_t side = plan.side_stream;
  cudaEventRecord(plan.ev_fork, stream);
  cudaStreamWaitEvent(side, plan.ev_fork, 0);
  if (copy_beside) {
    k_scaled_copy<Sreal, F><<<g2, 256, 0, side>>>(P, S, fb.scale, L, T, INT_MAX);
    cudaEventRecord(plan.ev_copy, side);
  }
  for (int kt = 0; kt < plan.nsteps; ++kt) {
    if (kt >= 2) cudaStreamWaitEvent(stream, plan.ev_update[kt - 2], 0);
    if (kt == 1 && copy_beside) cudaStreamWaitEvent(stream, plan.ev_copy, 0);
    const int npn = plan.h_panel_off[kt + 1] - plan.h_panel_off[kt];
    const int2* pitems = plan.panel_items + plan.h_panel_off[kt];
    bool stacked = true;
    if constexpr (sizeof(F) == 4 && T == 64) {
      if (plan.split) {   // diagonal tiles (factor + inverse), then the tiles below them
        stacked = false;
        const int nd = plan.h_diag_count[kt];
        if (nd > 0)
          launch_prio(k_chol_diag<F, T>, nd, DiagLayout<F, T>::bytes, stream, plan.prio_high, (const F*)L, Dinv, P,
                      pitems, kt, fb.fail_flags, fb.boosted, fb.v_total);
        if (npn > nd)
          launch_prio(k_chol_trsm<F, T>, npn - nd, TrsmLayout<F, T>::bytes, stream, plan.prio_high, L,
                      (const F*)Dinv, P, pitems + nd, kt, fb.v_total);
      }
    }
    if (stacked && npn > 0)
      launch_prio_n(k_chol_panel<F, T>, npn, PANEL_THREADS, panel_smem<F, T>(npn), stream, plan.prio_high, L,
                    reinterpret_cast<F*>(fb.Ldiag), P, pitems, kt, fb.fail_flags, fb.boosted);
    cudaEventRecord(plan.ev_panel[kt], stream);
    cudaStreamWaitEvent(side, plan.ev_panel[kt], 0);
    const int nu = plan.h_update_off[kt + 1] - plan.h_update_off[kt];
    if (nu > 0) {
      launch_prio(k_chol_update<F, T>, nu, 0, side, plan.prio_low, L, P, plan.update_items + plan.h_update_off[kt], kt);
    }
    cudaEventRecord(plan.ev_update[kt], side);
  }
  cudaEventRecord(plan.ev_join, side);
  cudaStreamWaitEvent(stream, plan.ev_join, 0);
  // the split panel's diagonal kernels wrote the inverses
  if (plan.n_diag_items > 0 && !plan.split)
    k_diag_inverse<F, T><<<plan.n_diag_items, 256, 0, stream>>>(reinterpret_cast<const F*>(fb.Ldiag), Dinv, P,
                                                                plan.diag_items, fb.v_total);
}

template <typename F, int T>
void launch_solve_t(const DevProblem& P, const double* S, const double* b, const FactorBuffers& fb,
                    const CholPlan& plan, int refine_steps, cudaStream_t stream) {
  using Sreal = double;
  const F* L = reinterpret_cast<const F*>(fb.L);
  const F* Dinv = reinterpret_cast<const F*>(fb.Dinv);
  for (int s = 0; s <= refine_steps; ++s) {   // x = S~^-1 b, then x += S~^-1 (b - S x)
    launch_tri_solve<F, T, Sreal>(P, L, Dinv, fb.scale, s ? fb.r : b, fb.x, s < refine_steps && s == 0 ? fb.r : nullptr,
                                  s > 0, plan.max_np, fb.v_total, plan.solve_cs, fb.fail_flags,
                                  s ? plan.n_res_items > 0 : tensor_steps<F, T>(plan), stream);
    if (s == refine_steps) break;
    if (s > 0) cudaMemcpyAsync(fb.r, b, (size_t)fb.v_total * sizeof(double), cudaMemcpyDeviceToDevice, stream);
    if (plan.n_res_items > 0) {
      if (s == 0)
        launch_after(chained(P), k_residual<Sreal>, plan.n_res_items, 32 * RES_WARPS, stream, P, S, fb.x, fb.r,
                     plan.res_items);
      else
        k_residual<Sreal><<<plan.n_res_items, 32 * RES_WARPS, 0, stream>>>(P, S, fb.x, fb.r, plan.res_items);
    }
  }
}

// the tile size of the plan: FP32 factors 32 or 64 (chosen by stba_autotune), FP64 factors 32
template <typename F>
void launch_factor(const DevProblem& P, const double* S, const FactorBuffers& fb, const CholPlan& plan,
                   cudaStream_t stream) {
  if constexpr (sizeof(F) == 4) {
    if (plan.tile == 64) return launch_factor_t<F, 64>(P, S, fb, plan, stream);
  }
  launch_factor_t<F, 32>(P, S, fb, plan, stream);
}

template <typename F>
void launch_solve(const DevProblem& P, const double* S, const double* b, const FactorBuffers& fb,
                  const CholPlan& plan, int refine_steps, cudaStream_t stream) {
  if constexpr (sizeof(F) == 4) {
    if (plan.tile == 64) return launch_solve_t<F, 64>(P, S, b, fb, plan, refine_steps, stream);
  }
  launch_solve_t<F, 32>(P, S, b, fb, plan, refine_steps, stream);
}

size_t solve_smem_bytes(bool mixed, int tile, int max_np) {   // with the smallest stage count
  if (!mixed) return solve_cta_bytes<double, 32>(2, max_np);
  return tile == 64 ? solve_cta_bytes<float, 64>(2, max_np) : solve_cta_bytes<float, 32>(2, max_np);
}

int num_sms() {
  if (g_num_sms <= 0) {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&g_num_sms, cudaDevAttrMultiProcessorCount, dev);
    if (g_num_sms <= 0) g_num_sms = 1;
  }
  return g_num_sms;
}

// The largest dynamic shared memory of a kernel is a per-function attribute shared by every context of the
// process.  It is only ever raised: a context with smaller clusters must not lower it below what another
// live context's next launch asks for.
static void raise_smem_attr(const void* fn, int bytes) {
  static std::mutex mu;
  static std::map<std::pair<int, const void*>, int> set_to;
  int dev = 0;
  cudaGetDevice(&dev);
  std::lock_guard<std::mutex> lock(mu);
  int& cur = set_to[{dev, fn}];
  if (bytes > cur && cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes) == cudaSuccess)
    cur = bytes;
}

void configure_solve_kernels(int max_np) {
  int dev = 0, per_sm = 0, reserved = 0, optin = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&per_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev);
  cudaDeviceGetAttribute(&reserved, cudaDevAttrReservedSharedMemoryPerBlock, dev);
  cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  cudaDeviceGetAttribute(&g_num_sms, cudaDevAttrMultiProcessorCount, dev);
  g_smem_optin = optin;
  const int spread = per_sm / 2 - reserved + 128;   // two CTAs asking this much exceed one SM
  g_panel_min_smem = (per_sm > 0 && spread > 0 && spread <= optin) ? (size_t)spread : 0;
  raise_smem_attr((const void*)k_chol_panel<float, 64>, (int)panel_smem<float, 64>());
  raise_smem_attr((const void*)k_chol_panel<float, 32>, (int)panel_smem<float, 32>());
  raise_smem_attr((const void*)k_chol_panel<double, 32>, (int)panel_smem<double, 32>());
  raise_smem_attr((const void*)k_step_tc<true>, (int)std::max(PTC_SMEM, TCU_SMEM));
  raise_smem_attr((const void*)k_step_tc<false>, (int)std::max(PTC_SMEM, TCU_SMEM));
  raise_smem_attr((const void*)k_chol_diag<float, 64>, (int)DiagLayout<float, 64>::bytes);
  raise_smem_attr((const void*)k_chol_trsm<float, 64>, (int)TrsmLayout<float, 64>::bytes);
  // room for three stages wherever solve_stages may choose them
  auto stages = [&](size_t three) { return three <= (size_t)optin ? 3 : 2; };
  const int f64 = stages(solve_cta_bytes<float, 64>(3, max_np)) * SolveLayout<float, 64>::stage_bytes +
                  sizeof(float) * max_np;
  const int f32 = stages(solve_cta_bytes<float, 32>(3, max_np)) * SolveLayout<float, 32>::stage_bytes +
                  sizeof(float) * max_np;
  const int d32 = stages(solve_cta_bytes<double, 32>(3, max_np)) * SolveLayout<double, 32>::stage_bytes +
                  sizeof(double) * max_np;
  auto push = [&](auto* kern, size_t bytes) {
    if (bytes <= (size_t)optin) raise_smem_attr((const void*)kern, (int)bytes);
  };
#define PUSH_ATTR(F, T, CS) push(k_tri_push<F, T, double, CS>, PushLayout<F, T>::bytes(max_np / T, CS))
  PUSH_ATTR(float, 64, 2);
  PUSH_ATTR(float, 64, 4);
  PUSH_ATTR(float, 64, 8);
  PUSH_ATTR(float, 32, 2);
  PUSH_ATTR(float, 32, 4);
  PUSH_ATTR(float, 32, 8);
  PUSH_ATTR(double, 32, 2);
  PUSH_ATTR(double, 32, 4);
  PUSH_ATTR(double, 32, 8);
#undef PUSH_ATTR
  raise_smem_attr((const void*)k_tri_solve<float, 64, double, 8>, f64);
  raise_smem_attr((const void*)k_tri_solve<float, 32, double, 8>, f32);
  raise_smem_attr((const void*)k_tri_solve<double, 32, double, 8>, d32);
  raise_smem_attr((const void*)k_tri_solve<float, 64, double, 4>, f64);
  raise_smem_attr((const void*)k_tri_solve<float, 32, double, 4>, f32);
  raise_smem_attr((const void*)k_tri_solve<double, 32, double, 4>, d32);
  raise_smem_attr((const void*)k_tri_solve<float, 64, double, 2>, f64);
  raise_smem_attr((const void*)k_tri_solve<float, 32, double, 2>, f32);
  raise_smem_attr((const void*)k_tri_solve<double, 32, double, 2>, d32);
}

template void launch_factor<float>(const DevProblem&, const double*, const FactorBuffers&, const CholPlan&,
                                   cudaStream_t);
template void launch_factor<double>(const DevProblem&, const double*, const FactorBuffers&, const CholPlan&,
                                    cudaStream_t);
template void launch_solve<float>(const DevProblem&, const double*, const double*, const FactorBuffers&,
                                  const CholPlan&, int, cudaStream_t);
template void launch_solve<double>(const DevProblem&, const double*, const double*, const FactorBuffers&,
                                   const CholPlan&, int, cudaStream_t);

}  // namespace stba
