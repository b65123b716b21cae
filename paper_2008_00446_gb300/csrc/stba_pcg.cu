// Comparator of the method: plain LM with the full reduced camera system of all cameras (Eq. 5-6,
// S dc = b, S = B - E C^-1 E^T with the physical points; no clusters), solved by block-Jacobi
// preconditioned conjugate gradients, matrix-free.
//
//   k_pcg_jac      per observation: J_c (2x9) and J_p (2x3) at the current x, stored once per LM iteration;
//                  k_pcg_slot_j copies them into the order of the camera passes' slots
//   k_pcg_precond  per camera (one warp per 32 of its observations): the diagonal block
//                  S_jj = B_jj - sum_o J_c^T J_p C^-1 J_p^T J_c (undamped B part), diag(J_c^T J_c) and
//                  v = -J_c^T f; k_pcg_invert adds lambda diag(B) and inverts S_jj (9x9 Cholesky, FP64)
//   S p            k_pcg_Et (per observation, segmented by point: t = E^T p), k_pcg_u (u = C^-1 t), then
//                  k_pcg_cam (per camera: y = sum_o J_c^T (J_c p_j - J_p u) + lambda diag(B) p_j)
//   CG vectors     one thread per entry (9 per camera; the 9x9 preconditioner through shared memory), FP64;
//                  the scalars alpha, beta and the residual norms stay on the device (k_pcg_update, k_pcg_dir).
// A CG iteration is five launches: E^T p, u, the camera pass (which also forms p.q), k_pcg_update, k_pcg_dir;
// each clears what the next iteration adds into (k_pcg_u: t; k_pcg_dir: q and p.q).  It is bound by the two
// reads of the Jacobians (2 x 96 bytes per observation), stored so that a warp reads 512 contiguous bytes per
// load in both orders: 1000 cameras, 1.1M observations, 204 -> 80 us per CG iteration (before: rows of 96
// bytes gathered in the camera pass, and every thread of k_pcg_update / k_pcg_dir summing 456 FP64 partials,
// 55 us each on the 1/64-rate FP64 pipe).
// The right-hand side b = v - E C^-1 w is S applied to nothing but the point part: k_pcg_cam with p = 0
// and u = C^-1 w.
//
// Split variant (STBA_SOLVER_PCG_CLUSTERS; Sec. 6, the inexact solve of the split RCS): the method's own
// clustered system S' dc = b' (Eq. 10, 13, virtual points, correction) solved by the same PCG instead of the
// cluster factorisations.  The camera pass provides b' and the diagonal blocks of S' (the preconditioner);
// S' p = B p - E' C'^-1 E'^T p runs over the virtual points (k_spcg_Et, k_spcg_u), and a virtual point with
// one observation enters through its cancellation-free form J_c^T (I + J_p L^-1 J_p^T)^-1 J_c (the camera
// pass's Woodbury form) (k_spcg_cam).  One CG runs over the block-diagonal system of all clusters at once
// (shared step lengths; its solution is every cluster's).
#include <climits>

#include "stba_camera.cuh"
#include "stba_camtab.cuh"
#include "stba_device.cuh"
#include "stba_internal.cuh"

namespace stba {

namespace {

constexpr int JSTRIDE = 24;   // J_c (18) + J_p (6) per observation, working precision
constexpr int PSTRIDE = 12;   // reals per camera of the working-precision direction p (9 used; 16-byte loads)
constexpr int PQ_SLOTS = 64;  // accumulators of p.q
constexpr int CAMS_PER_BLOCK = 32;
constexpr int VEC_THREADS = 9 * CAMS_PER_BLOCK;   // CG vectors: one thread per entry, 32 cameras per block

// 16-byte pieces of one record of J; record e is lane e % 32 of group e / 32, and a group's piece k is 32
// consecutive 16-byte words, so that a warp's access is 512 contiguous bytes.
template <typename real> struct JPieces {
  static constexpr int PER = 16 / (int)sizeof(real), N = JSTRIDE / PER;
};
template <typename real>
__device__ __forceinline__ size_t j_piece(size_t e, int k) {
  return ((e >> 5) * JPieces<real>::N + k) * 32 + (e & 31);
}
template <typename real>
__device__ __forceinline__ void store_j(real* J, size_t e, const real (&v)[JSTRIDE]) {
#pragma unroll
  for (int k = 0; k < JPieces<real>::N; ++k) {
    if constexpr (sizeof(real) == 4)
      reinterpret_cast<float4*>(J)[j_piece<real>(e, k)] = make_float4(v[4 * k], v[4 * k + 1], v[4 * k + 2], v[4 * k + 3]);
    else
      reinterpret_cast<double2*>(J)[j_piece<real>(e, k)] = make_double2(v[2 * k], v[2 * k + 1]);
  }
}
template <typename real>
__device__ __forceinline__ void load_j_vec(const real* __restrict__ J, size_t e, real (&v)[JSTRIDE]) {
#pragma unroll
  for (int k = 0; k < JPieces<real>::N; ++k) {
    if constexpr (sizeof(real) == 4) {
      const float4 t = __ldg(reinterpret_cast<const float4*>(J) + j_piece<real>(e, k));
      v[4 * k] = t.x;
      v[4 * k + 1] = t.y;
      v[4 * k + 2] = t.z;
      v[4 * k + 3] = t.w;
    } else {
      const double2 t = __ldg(reinterpret_cast<const double2*>(J) + j_piece<real>(e, k));
      v[2 * k] = t.x;
      v[2 * k + 1] = t.y;
    }
  }
}

template <typename real>
__global__ void __launch_bounds__(256) k_pcg_jac(DevProblem P, real* __restrict__ J) {
  for (int o = blockIdx.x * blockDim.x + threadIdx.x; o < P.q; o += gridDim.x * blockDim.x) {
    // the rows of the virtual-point and camera passes, bitwise: the products cancel against V' and the
    // diagonal blocks by up to 1 / lambda
    const int cam = P.obs_cam[o];
    const CamRow<real> C = gather_camrow<real>(P, cam);
    real X[3], r[2], Jc[2][9], Jp[2][3], Jl[9];
    load_point_w(P, P.obs_pt[o], X);
    proj_rows<real, true>(C, X, Jc, Jp);
    load_jl(P, cam, Jl);
    apply_jl<real>(Jl, Jc);
    r[0] = res_ptr<real>(P)[2 * (size_t)o];
    r[1] = res_ptr<real>(P)[2 * (size_t)o + 1];
    scale_rows(row_weight<real>(P, r[0], r[1]), r, Jc, Jp);   // robust loss: sqrt(rho') rows
    real v[JSTRIDE];
#pragma unroll
    for (int c = 0; c < 9; ++c) {
      v[c] = Jc[0][c];
      v[9 + c] = Jc[1][c];
    }
#pragma unroll
    for (int s = 0; s < 3; ++s) {
      v[18 + s] = Jp[0][s];
      v[21 + s] = Jp[1][s];
    }
    store_j(J, (size_t)o, v);
  }
}

// J in the order of the camera passes' slots (a padding slot's record is never written nor read)
template <typename real>
__global__ void __launch_bounds__(256) k_pcg_slot_j(CamSlots CS, const real* __restrict__ J, real* __restrict__ Js) {
  const size_t n = 32 * (size_t)CS.nwarps;
  for (size_t sl = blockIdx.x * (size_t)blockDim.x + threadIdx.x; sl < n; sl += (size_t)gridDim.x * blockDim.x) {
    const int o = CS.slots[sl];
    if (o < 0) continue;
    real v[JSTRIDE];
    load_j_vec(J, (size_t)o, v);
    store_j(Js, sl, v);
  }
}

template <typename real>
__device__ __forceinline__ void unpack_j(const real (&v)[JSTRIDE], real (&Jc)[2][9], real (&Jp)[2][3]) {
#pragma unroll
  for (int c = 0; c < 9; ++c) {
    Jc[0][c] = v[c];
    Jc[1][c] = v[9 + c];
  }
#pragma unroll
  for (int s = 0; s < 3; ++s) {
    Jp[0][s] = v[18 + s];
    Jp[1][s] = v[21 + s];
  }
}
template <typename real>
__device__ __forceinline__ void load_j(const real* J, size_t e, real (&Jc)[2][9], real (&Jp)[2][3]) {
  real v[JSTRIDE];
  load_j_vec(J, e, v);
  unpack_j(v, Jc, Jp);
}

// the 9 entries of camera j of p (16-byte aligned records of PSTRIDE reals)
template <typename real>
__device__ __forceinline__ void load_p9(const real* __restrict__ p, int j, real (&v)[9]) {
  const real* s = p + PSTRIDE * (size_t)j;
  if constexpr (sizeof(real) == 4) {
    const float4 a = *reinterpret_cast<const float4*>(s), b = *reinterpret_cast<const float4*>(s + 4);
    v[0] = a.x;
    v[1] = a.y;
    v[2] = a.z;
    v[3] = a.w;
    v[4] = b.x;
    v[5] = b.y;
    v[6] = b.z;
    v[7] = b.w;
    v[8] = s[8];
  } else {
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const double2 a = *reinterpret_cast<const double2*>(s + 2 * k);
      v[2 * k] = a.x;
      v[2 * k + 1] = a.y;
    }
    v[8] = s[8];
  }
}

// Sums over the warp of v[0..8]; lane i < 9 receives sum i.  Transposed: every step halves the values a lane holds, 16
// shuffles instead of 45.
template <typename real>
__device__ __forceinline__ real warp_sums9(const real (&v)[9]) {
  const int lane = threadIdx.x & 31;
  real x[8];
  const bool up = (lane & 8) != 0;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const real hi = i == 0 ? v[8] : real(0);
    x[i] = (up ? hi : v[i]) + __shfl_xor_sync(FULL_MASK, up ? v[i] : hi, 8);
  }
#pragma unroll
  for (int s = 4; s >= 1; s >>= 1) {
    const bool u = (lane & s) != 0;
#pragma unroll
    for (int i = 0; i < s; ++i) {
      const real send = u ? x[i] : x[i + s];
      x[i] = (u ? x[i + s] : x[i]) + __shfl_xor_sync(FULL_MASK, send, s);
    }
  }
  return x[0] + __shfl_xor_sync(FULL_MASK, x[0], 16);
}

// Per camera diagonal block of S (45 lower entries, without the damping), diag(B) and v = -J_c^T f.
template <typename real>
__global__ void __launch_bounds__(256) k_pcg_precond(DevProblem P, CamSlots CS, bool gather, const real* __restrict__ J,
                                                     const real* __restrict__ pt_info, double* __restrict__ Mblk,
                                                     double* __restrict__ Bdiag, real* __restrict__ vgrad) {
  const int gw = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (gw >= CS.nwarps) return;
  const int lane = threadIdx.x & 31;
  const int j = CS.warp_cam[gw];
  const int o = CS.slots[32 * (size_t)gw + lane];
  real Jc[2][9], Jp[2][3], f[2] = {0, 0};
  real H[3][9];   // C^-1 J_p^T J_c
#pragma unroll
  for (int c = 0; c < 9; ++c) Jc[0][c] = Jc[1][c] = H[0][c] = H[1][c] = H[2][c] = real(0);
#pragma unroll
  for (int s = 0; s < 3; ++s) Jp[0][s] = Jp[1][s] = real(0);
  if (o >= 0) {
    load_j(J, gather ? (size_t)o : 32 * (size_t)gw + lane, Jc, Jp);   // rows already scaled by sqrt(rho') under a robust loss
    f[0] = res_ptr<real>(P)[2 * (size_t)o];
    f[1] = res_ptr<real>(P)[2 * (size_t)o + 1];
    const real sw = huber_sqrt_weight<real>(P.huber_a, f[0], f[1]);
    f[0] *= sw;
    f[1] *= sw;
    const real* ci = pt_info + 9 * (size_t)CS.pv[32 * (size_t)gw + lane].x;   // C^-1 packed 00 01 02 11 12 22
    const real Ci[3][3] = {{ci[0], ci[1], ci[2]}, {ci[1], ci[3], ci[4]}, {ci[2], ci[4], ci[5]}};
#pragma unroll
    for (int c = 0; c < 9; ++c) {
      real g[3];
#pragma unroll
      for (int s = 0; s < 3; ++s) g[s] = Jp[0][s] * Jc[0][c] + Jp[1][s] * Jc[1][c];
#pragma unroll
      for (int s = 0; s < 3; ++s) H[s][c] = Ci[s][0] * g[0] + Ci[s][1] * g[1] + Ci[s][2] * g[2];
    }
  }
  // 45 + 9 + 9 terms, summed over the warp in two groups of 32 (transposed reduction)
  real sums[2];
#pragma unroll
  for (int half = 0; half < 2; ++half) {
    real v[32];
    int t = 0;
#pragma unroll
    for (int i = 0; i < 9; ++i)
#pragma unroll
      for (int jj = 0; jj <= i; ++jj, ++t) {
        if (t / 32 == half) {
          // (J_c^T J_c)_ij - (J_p^T J_c)_:i . H_:j
          real g0 = Jp[0][0] * Jc[0][i] + Jp[1][0] * Jc[1][i];
          real g1 = Jp[0][1] * Jc[0][i] + Jp[1][1] * Jc[1][i];
          real g2 = Jp[0][2] * Jc[0][i] + Jp[1][2] * Jc[1][i];
          v[t - 32 * half] = Jc[0][i] * Jc[0][jj] + Jc[1][i] * Jc[1][jj] - (g0 * H[0][jj] + g1 * H[1][jj] + g2 * H[2][jj]);
        }
      }
    if (half == 1) {
#pragma unroll
      for (int i = 0; i < 9; ++i) {
        v[45 - 32 + i] = Jc[0][i] * Jc[0][i] + Jc[1][i] * Jc[1][i];
        v[54 - 32 + i] = -(Jc[0][i] * f[0] + Jc[1][i] * f[1]);
      }
      v[31] = real(0);
    }
    // same transposed reduction as the camera pass
#pragma unroll
    for (int s = 16; s >= 1; s >>= 1) {
      const bool up = (lane & s) != 0;
#pragma unroll
      for (int i = 0; i < s; ++i) {
        const real send = up ? v[i] : v[i + s];
        const real keep = up ? v[i + s] : v[i];
        v[i] = keep + __shfl_xor_sync(FULL_MASK, send, s);
      }
    }
    sums[half] = v[0];
  }
#pragma unroll
  for (int half = 0; half < 2; ++half) {
    const int e = lane + 32 * half;
    if (e < 45)
      atomicAdd(Mblk + 45 * (size_t)j + e, (double)sums[half]);
    else if (e < 54)
      atomicAdd(Bdiag + 9 * (size_t)j + (e - 45), (double)sums[half]);
    else if (e < 63)
      atomicAdd(vgrad + 9 * (size_t)j + (e - 54), sums[half]);
  }
}

// Minv_j = (S_jj + lambda diag(B_j))^-1, dense 9x9 (row-major), FP64 Cholesky; a non-positive pivot falls back
// to the inverse of the damped diagonal.  One warp per camera: lane r < 9 holds row r of the matrix and of its
// factor in registers, a column's pivot and entries travel by shuffles; then lane c solves for column c of the
// inverse against the factor in shared memory.  (One thread per camera with the 9x9 arrays in local memory
// took 152 us for 1000 cameras.)
constexpr int INV_WARPS = 4;
__global__ void __launch_bounds__(32 * INV_WARPS) k_pcg_invert(int m, const double* __restrict__ Mblk,
                                                               const double* __restrict__ Bdiag, const DevState* st,
                                                               double* __restrict__ Minv) {
  __shared__ double Ls[INV_WARPS][9][9];
  const int j = blockIdx.x * INV_WARPS + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (j >= m) return;   // uniform per warp
  double(*L)[9] = Ls[threadIdx.x >> 5];
  const double lam = st->lambda_used;
  const int r = lane < 9 ? lane : 8;
  double A[9], d0 = 0.0;   // row r of the damped block (lower part), its diagonal entry
#pragma unroll
  for (int c = 0; c < 9; ++c) {
    A[c] = c <= r ? Mblk[45 * (size_t)j + r * (r + 1) / 2 + c] : 0.0;
    if (c == r) {
      A[c] += lam * Bdiag[9 * (size_t)j + r];
      d0 = A[c];
    }
  }
  bool ok = true;
#pragma unroll
  for (int c = 0; c < 9; ++c) {
    const double p = __shfl_sync(FULL_MASK, A[c], c);   // pivot
    ok = ok && p > 0.0;
    const double l = sqrt(ok ? p : 1.0);
    A[c] = r == c ? l : A[c] / l;   // column c of the factor (rows >= c)
#pragma unroll
    for (int k = c + 1; k < 9; ++k) A[k] -= A[c] * __shfl_sync(FULL_MASK, A[c], k);
  }
  double* out = Minv + 81 * (size_t)j;
  if (!ok) {   // uniform: every lane saw the same pivots
    if (lane < 9)
      for (int c = 0; c < 9; ++c) out[9 * lane + c] = (lane == c && d0 > 0.0) ? 1.0 / d0 : 0.0;
    return;
  }
  if (lane < 9) {
#pragma unroll
    for (int c = 0; c < 9; ++c) L[lane][c] = c <= lane ? A[c] : 0.0;
  }
  __syncwarp();
  if (lane < 9) {   // inverse = L^-T L^-1, column `lane`
    double y[9];
#pragma unroll
    for (int i = 0; i < 9; ++i) {
      double s = i == lane ? 1.0 : 0.0;
#pragma unroll
      for (int k = 0; k < i; ++k) s -= L[i][k] * y[k];
      y[i] = s / L[i][i];
    }
#pragma unroll
    for (int i = 8; i >= 0; --i) {
      double s = y[i];
#pragma unroll
      for (int k = i + 1; k < 9; ++k) s -= L[k][i] * y[k];
      y[i] = s / L[i][i];
    }
#pragma unroll
    for (int i = 0; i < 9; ++i) out[9 * i + lane] = y[i];
  }
}

// t_i = sum_{o in point i} J_p^T (J_c p_cam(o)), segmented by point (observations are sorted by point)
template <typename real>
__global__ void __launch_bounds__(256) k_pcg_Et(DevProblem P, const real* __restrict__ J, const real* __restrict__ p,
                                                real* __restrict__ t) {
  const int o = blockIdx.x * blockDim.x + threadIdx.x;
  const int lane = threadIdx.x & 31;
  const bool act = o < P.q;
  int pt = INT_MAX;
  real val[3] = {0, 0, 0};
  if (act) {
    pt = P.obs_pt[o];
    real Jc[2][9], Jp[2][3];
    load_j(J, (size_t)o, Jc, Jp);
    real pc[9];
    load_p9(p, P.obs_cam[o], pc);
    real a0 = 0, a1 = 0;
#pragma unroll
    for (int c = 0; c < 9; ++c) {
      a0 += Jc[0][c] * pc[c];
      a1 += Jc[1][c] * pc[c];
    }
#pragma unroll
    for (int s = 0; s < 3; ++s) val[s] = Jp[0][s] * a0 + Jp[1][s] * a1;
  }
  segmented_scan<3>(val, pt, lane);
  segmented_store<3>(val, pt, act, lane, o, P.pt_off, t);
}

// u_i = C_i^-1 t_i; clears t_i for the next E^T p
template <typename real>
__global__ void k_pcg_u(int n, const real* __restrict__ pt_info, real* __restrict__ t, real* __restrict__ u) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const real* ci = pt_info + 9 * (size_t)i;
    real* tp = t + 3 * (size_t)i;
    const real ti[3] = {tp[0], tp[1], tp[2]};
    real* ui = u + 3 * (size_t)i;
    ui[0] = ci[0] * ti[0] + ci[1] * ti[1] + ci[2] * ti[2];
    ui[1] = ci[1] * ti[0] + ci[3] * ti[1] + ci[4] * ti[2];
    ui[2] = ci[2] * ti[0] + ci[4] * ti[1] + ci[5] * ti[2];
    tp[0] = tp[1] = tp[2] = real(0);
  }
}

// Block sum of v over the first lanes of every warp, added to one of the PQ_SLOTS accumulators of p.q.
__device__ __forceinline__ void add_pq(double v, double* __restrict__ pq) {
  __shared__ double red[8];
#pragma unroll
  for (int d = 8; d > 0; d >>= 1) v += __shfl_xor_sync(FULL_MASK, v, d);   // lanes 0..15 (9 used)
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  if (threadIdx.x == 0) {
    double s = 0.0;
#pragma unroll
    for (int w = 0; w < 8; ++w) s += red[w];
    atomicAdd(pq + (blockIdx.x & (PQ_SLOTS - 1)), s);
  }
}

// The camera passes of a product: a warp takes `groups` consecutive groups of 32 slots (mostly of one camera),
// the next group's Jacobians in flight while it works on one; the sums of a group are added up in FP64 in lanes 0..8
// and go to memory once per camera.  Bound by the 96 bytes per observation of J (the previous product's other copy has
// displaced them from L2).  Per CG iteration of 1.1M observations / 280k observations: one group per warp and
// no prefetch 89 / 44 us; 4 groups 85 / 41, 8 groups 80 / 42, 2 resident CTAs (3: 85 / 45): 8 groups once they
// still leave 16 warps per SM, else 4.
static int cam_groups(int nwarps) { return nwarps >= 8 * 16 * num_sms() ? 8 : 4; }

// y_j += sum_{o in camera j} J_c^T (J_c p_j - J_p u_pt(o)) (+ lambda diag(B_j) p_j, added by the camera's first
// group), and pq += p.y.  With p = null the J_c p term is absent (right-hand side pass).
// GATHER: J is in observation order (there was no room for the copy in slot order).
template <typename real, bool GATHER>
__global__ void __launch_bounds__(256, sizeof(real) == 4 ? 2 : 1)
    k_pcg_cam(CamSlots CS, int groups, const real* __restrict__ J, const real* __restrict__ p,
              const double* __restrict__ pvec, const real* __restrict__ u, const double* __restrict__ Bdiag,
              const DevState* st, double* __restrict__ y, double* __restrict__ pq) {
  const int g0 = groups * ((blockIdx.x * blockDim.x + threadIdx.x) >> 5), g1 = min(g0 + groups, CS.nwarps);
  const int lane = threadIdx.x & 31;
  double dot = 0.0;
  if (g0 < g1) {
    real v[9], Jn[JSTRIDE];
    int pt_n = -1;   // point of the prefetched slot, -1 for a padding slot
    auto fetch = [&](int g) {
      const size_t sl = 32 * (size_t)g + lane;
      const int o = CS.slots[sl];
      // unconditional (a padding slot's record is unused): in slot order not behind the load of the slot
      load_j_vec(J, GATHER ? (size_t)max(o, 0) : sl, Jn);
      const int pt = CS.pv[sl].x;
      pt_n = o >= 0 ? pt : -1;
    };
    fetch(g0);
    bool first = g0 == 0 || CS.warp_cam[g0 - 1] != CS.warp_cam[g0];   // the camera's first group is this warp's
    double add = 0.0;
    for (int g = g0; g < g1; ++g) {
      const int j = CS.warp_cam[g];
      const int pt = pt_n;
      real Jc[2][9], Jp[2][3];
      unpack_j(Jn, Jc, Jp);
      if (g + 1 < g1) fetch(g + 1);
#pragma unroll
      for (int c = 0; c < 9; ++c) v[c] = real(0);
      if (pt >= 0) {
        const real* ui = u + 3 * (size_t)pt;
        real a0 = -(Jp[0][0] * ui[0] + Jp[0][1] * ui[1] + Jp[0][2] * ui[2]);
        real a1 = -(Jp[1][0] * ui[0] + Jp[1][1] * ui[1] + Jp[1][2] * ui[2]);
        if (p) {
          real pj[9];
          load_p9(p, j, pj);
#pragma unroll
          for (int c = 0; c < 9; ++c) {
            a0 += Jc[0][c] * pj[c];
            a1 += Jc[1][c] * pj[c];
          }
        }
#pragma unroll
        for (int c = 0; c < 9; ++c) v[c] = Jc[0][c] * a0 + Jc[1][c] * a1;
      }
      add += (double)warp_sums9(v);
      const int jn = g + 1 < g1 ? CS.warp_cam[g + 1] : -1;
      if (jn != j) {   // the camera's last group of this warp
        if (lane < 9) {
          if (p) {
            if (first) add += st->lambda_used * Bdiag[9 * (size_t)j + lane] * (double)p[PSTRIDE * (size_t)j + lane];
            dot += add * pvec[9 * (size_t)j + lane];
          }
          atomicAdd(y + 9 * (size_t)j + lane, add);
        }
        add = 0.0;
        first = true;
      }
    }
  }
  if (p) add_pq(dot, pq);
}

// split variant: zero the diagonal blocks of S' before the camera pass accumulates into them
__global__ void k_spcg_zero(DevProblem P, double* __restrict__ S) {
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < 81 * P.m; e += gridDim.x * blockDim.x) {
    const int j = e / 81, rc = e - 81 * (e / 81), r = rc / 9, c = rc - 9 * (rc / 9);
    const int k = P.cam_cluster[j], lc = P.cam_local[j], np = P.cluster_np[k];
    S[P.S_off[k] + (size_t)(9 * lc + r) * np + 9 * lc + c] = 0.0;
  }
}

// split variant: the damped diagonal blocks of S' (45 lower entries) and b' of every camera, from the
// cluster layout filled by the camera pass
__global__ void k_spcg_blocks(DevProblem P, const double* __restrict__ S, const double* __restrict__ b,
                              double* __restrict__ Mblk, double* __restrict__ rhs) {
  for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < P.m; j += gridDim.x * blockDim.x) {
    const int k = P.cam_cluster[j], lc = P.cam_local[j], np = P.cluster_np[k];
    const double* Sk = S + P.S_off[k] + (size_t)(9 * lc) * np + 9 * lc;
    int t = 0;
    for (int r = 0; r < 9; ++r)
      for (int c = 0; c <= r; ++c, ++t) Mblk[45 * (size_t)j + t] = Sk[(size_t)r * np + c];
    for (int r = 0; r < 9; ++r) rhs[9 * (size_t)j + r] = b[P.v_off[k] + 9 * lc + r];
  }
}

// t_v = sum_{o in v} J_p^T (J_c p_cam(o)), segmented by virtual point
template <typename real>
__global__ void __launch_bounds__(256) k_spcg_Et(DevProblem P, const real* __restrict__ J, const real* __restrict__ p,
                                                 real* __restrict__ t) {
  const int o = blockIdx.x * blockDim.x + threadIdx.x;
  const int lane = threadIdx.x & 31;
  const bool act = o < P.q;
  int v = INT_MAX;
  real val[3] = {0, 0, 0};
  if (act) {
    v = P.obs_vp[o];
    real Jc[2][9], Jp[2][3];
    load_j(J, (size_t)o, Jc, Jp);
    real pc[9];
    load_p9(p, P.obs_cam[o], pc);
    real a0 = 0, a1 = 0;
#pragma unroll
    for (int c = 0; c < 9; ++c) {
      a0 += Jc[0][c] * pc[c];
      a1 += Jc[1][c] * pc[c];
    }
#pragma unroll
    for (int s = 0; s < 3; ++s) val[s] = Jp[0][s] * a0 + Jp[1][s] * a1;
  }
  segmented_scan<3>(val, v, lane);
  segmented_store<3>(val, v, act, lane, o, P.vp_off, t);
}

// u_v = V'_v^-1 t_v with V' = L L^T (L^-1 packed in vp_info), clearing t_v; nv from the device counter
template <typename real>
__global__ void k_spcg_u(const long long* __restrict__ counts, const real* __restrict__ vp_info,
                         real* __restrict__ t, real* __restrict__ u) {
  const long long nv = counts[0];
  for (long long v = blockIdx.x * (long long)blockDim.x + threadIdx.x; v < nv; v += (long long)gridDim.x * blockDim.x) {
    real Li[6], tv[3], uv[3];
#pragma unroll
    for (int c = 0; c < 6; ++c) Li[c] = vp_info[VPI * v + c];
#pragma unroll
    for (int c = 0; c < 3; ++c) tv[c] = t[3 * v + c];
    chol3_apply(Li, tv, uv);
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      u[3 * v + c] = uv[c];
      t[3 * v + c] = real(0);
    }
  }
}

// y_j += sum over the camera's observations of J_c^T N J_c p_j (single-observation virtual points, N =
// (I + J_p Lambda^-1 J_p^T)^-1, Lambda = lambda diag(J_p^T J_p)) or J_c^T (J_c p_j - J_p u_v) (the others),
// plus lambda diag(J_c^T J_c) p_j: S' p for the cameras of every cluster
template <typename real, bool GATHER>
__global__ void __launch_bounds__(256, sizeof(real) == 4 ? 2 : 1)
    k_spcg_cam(CamSlots CS, int groups, const real* __restrict__ J, const real* __restrict__ p,
               const double* __restrict__ pvec, const real* __restrict__ u, const DevState* st,
               double* __restrict__ y, double* __restrict__ pq) {
  const int g0 = groups * ((blockIdx.x * blockDim.x + threadIdx.x) >> 5), g1 = min(g0 + groups, CS.nwarps);
  const int lane = threadIdx.x & 31;
  const real lam = (real)st->lambda_used;
  double dot = 0.0;
  if (g0 < g1) {
    real vsum[9], Jn[JSTRIDE];
    int vs_n = 0;       // virtual point of the prefetched slot, bit 31: it has no other observation
    bool act_n = false;   // not a padding slot
    auto fetch = [&](int g) {
      const size_t sl = 32 * (size_t)g + lane;
      const int o = CS.slots[sl];
      load_j_vec(J, GATHER ? (size_t)max(o, 0) : sl, Jn);   // as in k_pcg_cam
      vs_n = CS.pv[sl].y;
      act_n = o >= 0;
    };
    fetch(g0);
    double add = 0.0;
    for (int g = g0; g < g1; ++g) {
      const int j = CS.warp_cam[g];
      const int vs = vs_n;
      const bool act = act_n;
      real Jc[2][9], Jp[2][3];
      unpack_j(Jn, Jc, Jp);
      if (g + 1 < g1) fetch(g + 1);
#pragma unroll
      for (int c = 0; c < 9; ++c) vsum[c] = real(0);
      if (act) {
        real pj[9];
        load_p9(p, j, pj);
        real a0 = 0, a1 = 0;
#pragma unroll
        for (int c = 0; c < 9; ++c) {
          a0 += Jc[0][c] * pj[c];
          a1 += Jc[1][c] * pj[c];
        }
        real b0, b1;
        if (vs < 0) {
          real K00 = 0, K01 = 0, K11 = 0;
#pragma unroll
          for (int s = 0; s < 3; ++s) {
            const real il = real(1) / (lam * (Jp[0][s] * Jp[0][s] + Jp[1][s] * Jp[1][s]));
            K00 += Jp[0][s] * Jp[0][s] * il;
            K01 += Jp[0][s] * Jp[1][s] * il;
            K11 += Jp[1][s] * Jp[1][s] * il;
          }
          const real idet = real(1) / ((real(1) + K00) * (real(1) + K11) - K01 * K01);
          b0 = ((real(1) + K11) * a0 - K01 * a1) * idet;
          b1 = (-K01 * a0 + (real(1) + K00) * a1) * idet;
        } else {
          const real* uv = u + 3 * (size_t)vs;
          b0 = a0 - (Jp[0][0] * uv[0] + Jp[0][1] * uv[1] + Jp[0][2] * uv[2]);
          b1 = a1 - (Jp[1][0] * uv[0] + Jp[1][1] * uv[1] + Jp[1][2] * uv[2]);
        }
#pragma unroll
        for (int c = 0; c < 9; ++c)
          vsum[c] = Jc[0][c] * b0 + Jc[1][c] * b1 + lam * (Jc[0][c] * Jc[0][c] + Jc[1][c] * Jc[1][c]) * pj[c];
      }
      add += (double)warp_sums9(vsum);
      const int jn = g + 1 < g1 ? CS.warp_cam[g + 1] : -1;
      if (jn != j) {
        if (lane < 9) {
          dot += add * pvec[9 * (size_t)j + lane];
          atomicAdd(y + 9 * (size_t)j + lane, add);
        }
        add = 0.0;
      }
    }
  }
  add_pq(dot, pq);
}

// Block sum (VEC_THREADS threads) of N per-thread values, returned to every thread (fixed order).
template <int N>
__device__ __forceinline__ void block_sums(double (&v)[N]) {
  __shared__ double red[N][VEC_THREADS / 32];
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
  for (int i = 0; i < N; ++i) {
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) v[i] += __shfl_xor_sync(FULL_MASK, v[i], d);
    if (lane == 0) red[i][w] = v[i];
  }
  __syncthreads();
#pragma unroll
  for (int i = 0; i < N; ++i) {
    double s = 0.0;
#pragma unroll
    for (int k = 0; k < VEC_THREADS / 32; ++k) s += red[i][k];
    v[i] = s;
  }
  __syncthreads();
}

// z = (Minv_j r_j)[a] for thread t = 9 (j - j0) + a of the block's 32 cameras; rs holds their r
__device__ __forceinline__ double apply_minv_row(const double* __restrict__ Minv, size_t i, const double* rs, int t) {
  const double* M = Minv + 9 * i;   // row a of camera j: 81 j + 9 a = 9 i
  const double* r = rs + 9 * (t / 9);
  double s = 0.0;
#pragma unroll
  for (int b = 0; b < 9; ++b) s += M[b] * r[b];
  return s;
}

// r = b (= v + y from the right-hand-side pass), x = 0, z = Minv r, p = z; y = 0 for the first product;
// partials of r.z and r.r
template <typename real>
__global__ void __launch_bounds__(VEC_THREADS) k_pcg_init(int m, const real* __restrict__ vgrad,
                                                          double* __restrict__ yrhs, const double* __restrict__ Minv,
                                                          double* x, double* r, double* pvec, real* pw,
                                                          double* partial) {
  __shared__ double rs[VEC_THREADS];
  const int t = threadIdx.x;
  double sums[2] = {0, 0};
  for (int j0 = blockIdx.x * CAMS_PER_BLOCK; j0 < m; j0 += gridDim.x * CAMS_PER_BLOCK) {
    const size_t i = 9 * (size_t)j0 + t;
    const bool act = i < 9 * (size_t)m;
    double ri = 0.0;
    if (act) {
      ri = (vgrad ? (double)vgrad[i] : 0.0) + yrhs[i];
      yrhs[i] = 0.0;
      x[i] = 0.0;
      r[i] = ri;
    }
    rs[t] = ri;
    __syncthreads();
    if (act) {
      const double z = apply_minv_row(Minv, i, rs, t);
      pvec[i] = z;
      pw[PSTRIDE * (size_t)(j0 + t / 9) + t % 9] = (real)z;
      sums[0] += ri * z;
      sums[1] += ri * ri;
    }
    __syncthreads();
  }
  block_sums(sums);
  if (t == 0) {
    partial[blockIdx.x] = sums[0];
    partial[RED_BLOCKS + blockIdx.x] = sums[1];
  }
}

// sums of the nb partials of r.z and r.r, the same in every block
__device__ __forceinline__ void sum_partials2(const double* __restrict__ partial, int nb, double (&s)[2]) {
  s[0] = s[1] = 0.0;
  for (int i = threadIdx.x; i < nb; i += VEC_THREADS) {
    s[0] += partial[i];
    s[1] += partial[RED_BLOCKS + i];
  }
  block_sums(s);
}

// scalars: s[0] = b.b, s[1 + parity] = r.z, s[3] = r.r
__global__ void __launch_bounds__(VEC_THREADS) k_pcg_start(const double* partial, int nb, double* s) {
  double v[2];
  sum_partials2(partial, nb, v);
  if (threadIdx.x == 0) {
    s[1] = v[0];
    s[2] = 0.0;
    s[3] = v[1];
    s[0] = v[1];
  }
}

// alpha = r.z / p.q; x += alpha p; r -= alpha q; z = Minv r; partials of the new r.z and r.r
__global__ void __launch_bounds__(VEC_THREADS) k_pcg_update(int m, const double* __restrict__ pq_slots,
                                                            const double* __restrict__ s, int parity,
                                                            const double* __restrict__ pvec,
                                                            const double* __restrict__ q,
                                                            const double* __restrict__ Minv, double* x, double* r,
                                                            double* z, double* partial) {
  __shared__ double rs[VEC_THREADS];
  const int t = threadIdx.x;
  double pq[1] = {t < PQ_SLOTS ? pq_slots[t] : 0.0};
  block_sums(pq);
  const double alpha = (pq[0] != 0.0) ? s[1 + parity] / pq[0] : 0.0;
  double sums[2] = {0, 0};
  for (int j0 = blockIdx.x * CAMS_PER_BLOCK; j0 < m; j0 += gridDim.x * CAMS_PER_BLOCK) {
    const size_t i = 9 * (size_t)j0 + t;
    const bool act = i < 9 * (size_t)m;
    double ri = 0.0;
    if (act) {
      x[i] += alpha * pvec[i];
      ri = r[i] - alpha * q[i];
      r[i] = ri;
    }
    rs[t] = ri;
    __syncthreads();
    if (act) {
      const double zi = apply_minv_row(Minv, i, rs, t);
      z[i] = zi;
      sums[0] += ri * zi;
      sums[1] += ri * ri;
    }
    __syncthreads();
  }
  block_sums(sums);
  if (t == 0) {
    partial[blockIdx.x] = sums[0];
    partial[RED_BLOCKS + blockIdx.x] = sums[1];
  }
}

// beta = r.z_new / r.z_old; p = z + beta p (and its working-precision copy); the new scalars go to the
// other parity slot; q and the p.q accumulators are cleared for the next product
template <typename real>
__global__ void __launch_bounds__(VEC_THREADS) k_pcg_dir(int m9, const double* __restrict__ partial, int nb, double* s,
                                                         int parity, const double* __restrict__ z, double* pvec,
                                                         real* pw, double* q, double* pq_slots) {
  double v[2];
  sum_partials2(partial, nb, v);
  const double rz_old = s[1 + parity];
  const double beta = (rz_old != 0.0) ? v[0] / rz_old : 0.0;
  for (int i = blockIdx.x * VEC_THREADS + threadIdx.x; i < m9; i += gridDim.x * VEC_THREADS) {
    const double pn = z[i] + beta * pvec[i];
    pvec[i] = pn;
    pw[PSTRIDE * (size_t)(i / 9) + i % 9] = (real)pn;
    q[i] = 0.0;
  }
  if (blockIdx.x == 0) {
    if (threadIdx.x < PQ_SLOTS) pq_slots[threadIdx.x] = 0.0;
    if (threadIdx.x == 0) {
      s[1 + (1 - parity)] = v[0];
      s[3] = v[1];
    }
  }
}

__global__ void k_pcg_finish(int m9, const double* __restrict__ x, double* dc) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < m9; i += gridDim.x * blockDim.x) dc[i] = x[i];
}

// u_i = C_i^-1 w_i (the point part of the right-hand side; w is stored after C^-1 in pt_info)
template <typename real>
__global__ void k_pcg_uw(int n, const real* __restrict__ pt_info, real* __restrict__ u) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const real* ci = pt_info + 9 * (size_t)i;
    real* ui = u + 3 * (size_t)i;
    ui[0] = ci[0] * ci[6] + ci[1] * ci[7] + ci[2] * ci[8];
    ui[1] = ci[1] * ci[6] + ci[3] * ci[7] + ci[4] * ci[8];
    ui[2] = ci[2] * ci[6] + ci[4] * ci[7] + ci[5] * ci[8];
  }
}

}  // namespace

template <typename real>
void pcg_prepare(const DevProblem& P, Scratch<real> W, CamSlots CS, const PcgBuffers& B, DevState* st,
                 cudaStream_t stream) {
  const int m = P.m, m9 = 9 * P.m;
  real* J = reinterpret_cast<real*>(B.J);
  real* Js = reinterpret_cast<real*>(B.Jslot);
  real* pw = reinterpret_cast<real*>(B.pw);
  real* upt = reinterpret_cast<real*>(B.upt);
  const int obs_blocks = std::min((P.q + 255) / 256, num_sms() * 16);
  const int cam_blocks = (CS.nwarps + 7) / 8, groups = cam_groups(CS.nwarps);
  const int pt_blocks = std::min((P.n + 255) / 256, 4096);
  const int vec_blocks = std::min((m + CAMS_PER_BLOCK - 1) / CAMS_PER_BLOCK, RED_BLOCKS);
  k_pcg_jac<real><<<obs_blocks, 256, 0, stream>>>(P, J);
  if (Js) k_pcg_slot_j<real><<<std::min(cam_blocks, num_sms() * 16), 256, 0, stream>>>(CS, J, Js);
  cudaMemsetAsync(B.Bdiag, 0, 9 * (size_t)m * sizeof(double), stream);
  cudaMemsetAsync(B.pq, 0, PQ_SLOTS * sizeof(double), stream);
  const int inv_blocks = (m + INV_WARPS - 1) / INV_WARPS;
  if (B.split) {
    // the camera pass has filled the diagonal blocks of S' (damped) and b'
    launch_zero_vp3(B.tvp, B.counts, (int)sizeof(real), stream);
    k_spcg_blocks<<<(m + 127) / 128, 128, 0, stream>>>(P, W.S, W.b, B.Mblk, B.q);
    k_pcg_invert<<<inv_blocks, 32 * INV_WARPS, 0, stream>>>(m, B.Mblk, B.Bdiag, st, B.Minv);   // Bdiag = 0: no more damping
    k_pcg_init<real><<<vec_blocks, VEC_THREADS, 0, stream>>>(m, nullptr, B.q, B.Minv, B.x, B.r, B.p, pw, B.partial);
    k_pcg_start<<<1, VEC_THREADS, 0, stream>>>(B.partial, vec_blocks, B.scal);
    return;
  }
  cudaMemsetAsync(B.Mblk, 0, 45 * (size_t)m * sizeof(double), stream);
  cudaMemsetAsync(W.vgrad, 0, 9 * (size_t)m * sizeof(real), stream);
  cudaMemsetAsync(B.tpt, 0, 3 * (size_t)P.n * sizeof(real), stream);
  k_pcg_precond<real><<<cam_blocks, 256, 0, stream>>>(P, CS, !Js, Js ? Js : J, W.pt_info, B.Mblk, B.Bdiag, W.vgrad);
  k_pcg_invert<<<inv_blocks, 32 * INV_WARPS, 0, stream>>>(m, B.Mblk, B.Bdiag, st, B.Minv);
  // right-hand side b = v - E C^-1 w: the camera pass with p = 0 and u = C^-1 w
  k_pcg_uw<real><<<pt_blocks, 256, 0, stream>>>(P.n, W.pt_info, upt);
  cudaMemsetAsync(B.q, 0, (size_t)m9 * sizeof(double), stream);
  const auto pcg_cam = Js ? k_pcg_cam<real, false> : k_pcg_cam<real, true>;
  pcg_cam<<<(cam_blocks + groups - 1) / groups, 256, 0, stream>>>(CS, groups, Js ? Js : J, nullptr, nullptr, upt,
                                                                  B.Bdiag, st, B.q, B.pq);
  k_pcg_init<real><<<vec_blocks, VEC_THREADS, 0, stream>>>(m, W.vgrad, B.q, B.Minv, B.x, B.r, B.p, pw, B.partial);
  k_pcg_start<<<1, VEC_THREADS, 0, stream>>>(B.partial, vec_blocks, B.scal);
}

void launch_spcg_zero(const DevProblem& P, double* S, cudaStream_t stream) {
  k_spcg_zero<<<std::min((81 * P.m + 255) / 256, 4 * RED_BLOCKS), 256, 0, stream>>>(P, S);
}

template <typename real>
int pcg_iterate(const DevProblem& P, Scratch<real> W, CamSlots CS, const PcgBuffers& B, int max_iter, double tol,
                DevState* st, cudaStream_t stream) {
  const int m = P.m, m9 = 9 * P.m;
  real* J = reinterpret_cast<real*>(B.J);
  real* Js = reinterpret_cast<real*>(B.Jslot);
  real* pw = reinterpret_cast<real*>(B.pw);
  real* tpt = reinterpret_cast<real*>(B.tpt);
  real* upt = reinterpret_cast<real*>(B.upt);
  const int seg_blocks = (P.q + 255) / 256;
  const int cam_blocks = (CS.nwarps + 7) / 8, groups = cam_groups(CS.nwarps);
  const int pt_blocks = std::min((P.n + 255) / 256, 4096);
  const int vec_blocks = std::min((m + CAMS_PER_BLOCK - 1) / CAMS_PER_BLOCK, RED_BLOCKS);
  const auto pcg_cam = Js ? k_pcg_cam<real, false> : k_pcg_cam<real, true>;
  const auto spcg_cam = Js ? k_spcg_cam<real, false> : k_spcg_cam<real, true>;
  const real* Jc = Js ? Js : J;   // the camera passes' rows
  int it = 0;
  const double tol2 = tol * tol;
  // The GPU idles about 25 us at each reading of the residual (copy, synchronisation, the next launches); a solve
  // runs on average half an interval past its tolerance.  An interval of 8 took 4400 us (48 products) instead of 4180
  // (44) for a step of 1000 cameras (full system), 2240 instead of 2330 (48 both) for one of 500 cameras (split), and
  // twice the products wherever four are enough.
  constexpr int CHECK_EVERY = 4;
  while (it < max_iter) {
    const int upto = std::min(it + CHECK_EVERY, max_iter);
    for (; it < upto; ++it) {
      const int parity = it & 1;
      // q = S p and p.q
      if (B.split) {   // S' p over the virtual points
        real* tvp = reinterpret_cast<real*>(B.tvp);
        real* uvp = reinterpret_cast<real*>(B.uvp);
        k_spcg_Et<real><<<seg_blocks, 256, 0, stream>>>(P, J, pw, tvp);
        k_spcg_u<real><<<2 * RED_BLOCKS, 256, 0, stream>>>(B.counts, W.vp_info, tvp, uvp);
        spcg_cam<<<(cam_blocks + groups - 1) / groups, 256, 0, stream>>>(CS, groups, Jc, pw, B.p, uvp, st, B.q, B.pq);
      } else {
        k_pcg_Et<real><<<seg_blocks, 256, 0, stream>>>(P, J, pw, tpt);
        k_pcg_u<real><<<pt_blocks, 256, 0, stream>>>(P.n, W.pt_info, tpt, upt);
        pcg_cam<<<(cam_blocks + groups - 1) / groups, 256, 0, stream>>>(CS, groups, Jc, pw, B.p, upt, B.Bdiag, st, B.q,
                                                                        B.pq);
      }
      k_pcg_update<<<vec_blocks, VEC_THREADS, 0, stream>>>(m, B.pq, B.scal, parity, B.p, B.q, B.Minv, B.x, B.r, B.z,
                                                           B.partial);
      k_pcg_dir<real><<<vec_blocks, VEC_THREADS, 0, stream>>>(m9, B.partial, vec_blocks, B.scal, parity, B.z, B.p, pw,
                                                              B.q, B.pq);
    }
    double hs[4];
    if (cudaMemcpyAsync(hs, B.scal, sizeof hs, cudaMemcpyDeviceToHost, stream) != cudaSuccess ||
        cudaStreamSynchronize(stream) != cudaSuccess)
      break;
    if (!(hs[3] > tol2 * hs[0])) break;   // converged (or the residual is not finite)
  }
  k_pcg_finish<<<std::min((m9 + RED_THREADS - 1) / RED_THREADS, RED_BLOCKS), RED_THREADS, 0, stream>>>(m9, B.x, W.dc);
  launch_step_rows<real>(P, W.dc, W.edc, stream);
  return it;
}

#define PCG_INSTANTIATE(real)                                                                                  \
  template void pcg_prepare<real>(const DevProblem&, Scratch<real>, CamSlots, const PcgBuffers&, DevState*,   \
                                  cudaStream_t);                                                              \
  template int pcg_iterate<real>(const DevProblem&, Scratch<real>, CamSlots, const PcgBuffers&, int, double,  \
                                 DevState*, cudaStream_t);
PCG_INSTANTIATE(float)
PCG_INSTANTIATE(double)

}  // namespace stba
