// Per-iteration kernels of the STBA LM step (Algorithm 1), except the dense cluster factorisation.
//
//   k_begin          the state, the camera tables (stba_camtab.cuh), FP32 copies and the zeros of an iteration.
//   k_vp_reduce      per observation, warp-segmented by virtual point: V = sum Jp^T Jp, w' = -sum Jp^T f
//                    (Eq. 10: C' and w' of the split points).
//   k_pt_acc         per point (a warp per 32 points): C and w of the physical point, summed over its
//                    virtual points.
//   k_vp_finalize    per virtual point: steepest-descent correction of w' (Sec. 4.3, closed form below),
//                    damped V', its Cholesky inverse, y = V'^-1 w'; per point: physical C^-1 and w (Eq. 4)
//                    for Eq. 15.
//   k_cam_pass       per camera (a warp per 32 of its observations): the diagonal blocks of S'_k, b' and the
//                    camera gradient (Eq. 10/13).
//   k_pair_build     per camera pair of the camera graph inside a cluster: the off-diagonal blocks of S'_k.
//   k_scatter_step   dc in the cameras' order from the cluster solves, E dc, failed clusters.
//   k_point_rhs      per observation, warp-segmented by point: sum_o Jp^T Jc dc.
//   k_point_update   per point: dp = C^-1 (w - E^T dc) (Eq. 6 = Eq. 15), sums of the stop tests.
//   k_cost_cams, k_cost(_df)   F(x + dx) with FP64 sums; k_finalize: stop tests and the accept rule of Algorithm 1.
//
// Correction closed form: A has no camera columns and H~ = diag(H_lambda) is diagonal, so
// nu = (A H~^-1 A^T)^-1 A H~^-1 g makes H~^-1 (g - A^T nu) the H~-weighted projection of H~^-1 g on the
// steps where all virtual copies of a point are equal.  Per point and coordinate a:
//   dbar_a = sum_k w'_k,a / sum_k H~_k,a,  corrected w'_k,a = H~_k,a dbar_a,
// with H~_k = (1 + lambda) diag(V_k); the factor (1 + lambda) cancels.
#include <cfloat>
#include <climits>

#include "stba_camera.cuh"
#include "stba_camtab.cuh"
#include "stba_device.cuh"
#include "stba_strict.cuh"
#include "stba_internal.cuh"

namespace stba {

// ------------------------------------------------------------------------------------------------------
__device__ __forceinline__ void reset_state(DevState* st, const Settings& s) {
  st->lambda_used = st->lambda;
  st->corrected = (s.correction && st->lambda >= s.correction_lambda) ? 1 : 0;
  st->grad_max_bits = 0ull;
  st->failed = 0;
  st->nonfinite = 0;
  st->boosted = 0;
  st->pair_next = 0;
}

// the state alone, for the cost at x (an iteration resets it in k_begin)
__global__ void k_iter_begin(DevState* st, Settings s) {
  if (threadIdx.x == 0 && blockIdx.x == 0) reset_state(st, s);
}

void launch_iter_begin(DevState* st, const Settings& s, cudaStream_t stream) { k_iter_begin<<<1, 32, 0, stream>>>(st, s); }

// ------------------------------------------------------------------------------------------------------
template <typename real>
__global__ void __launch_bounds__(256) k_vp_reduce(DevProblem P, real* vp_acc) {
  chain_begin();
  const int o = blockIdx.x * blockDim.x + threadIdx.x;
  const int lane = threadIdx.x & 31;
  // sharded: only the observations of this process's clusters (a virtual point lies in one cluster, so its
  // observations are all in or all out)
  const bool act = o < P.q && (!P.sharded || P.cluster_owned[P.cam_cluster[P.obs_cam[o]]]);
  int v = INT_MAX;
  real val[9];
#pragma unroll
  for (int c = 0; c < 9; ++c) val[c] = 0;
  if (act) {
    v = P.obs_vp[o];
    const int cam = P.obs_cam[o];
    const int pt = P.vp_point[v];
    const CamRow<real> C = gather_camrow<real>(P, cam);
    real X[3];
    load_point_w(P, pt, X);
    real r[2], Jt[2][9], Jp[2][3];
    proj_rows<real, false>(C, X, Jt, Jp);
    r[0] = res_ptr<real>(P)[2 * (size_t)o];
    r[1] = res_ptr<real>(P)[2 * (size_t)o + 1];
    real sw;   // 1 without a robust loss
    if constexpr (sizeof(real) == 4)
      sw = huber_sqrt_weight_strict(P.huber_a, r[0], r[1]);
    else
      sw = huber_sqrt_weight<real>(P.huber_a, r[0], r[1]);
    r[0] *= sw;
    r[1] *= sw;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      Jp[0][c] *= sw;
      Jp[1][c] *= sw;
    }
    val[0] = Jp[0][0] * Jp[0][0] + Jp[1][0] * Jp[1][0];
    val[1] = Jp[0][0] * Jp[0][1] + Jp[1][0] * Jp[1][1];
    val[2] = Jp[0][0] * Jp[0][2] + Jp[1][0] * Jp[1][2];
    val[3] = Jp[0][1] * Jp[0][1] + Jp[1][1] * Jp[1][1];
    val[4] = Jp[0][1] * Jp[0][2] + Jp[1][1] * Jp[1][2];
    val[5] = Jp[0][2] * Jp[0][2] + Jp[1][2] * Jp[1][2];
#pragma unroll
    for (int j = 0; j < 3; ++j) val[6 + j] = -(Jp[0][j] * r[0] + Jp[1][j] * r[1]);
  }
  segmented_scan<9>(val, v, lane);
  segmented_store<9>(val, v, act, lane, o, P.vp_off, vp_acc);
}

template <typename real>
void launch_vp_reduce(const DevProblem& P, Scratch<real> W, cudaStream_t stream) {
  int blocks = (P.q + 255) / 256;
  launch_after(chained(P), k_vp_reduce<real>, blocks, 256, stream, P, W.vp_acc);
}

// ------------------------------------------------------------------------------------------------------
// FP64 arithmetic runs at 2 lanes a cycle and SM here, so a warp's FP64 instruction costs 16 cycles however few
// of its lanes matter, and shuffle trees in every warp of a CTA add up (8 warps x 5 steps: 640 cycles a value).
// The reductions below keep the tree in as few warps as possible, and maxima in the integer pipe: values >= 0
// order like their bits.
__device__ __forceinline__ unsigned long long warp_max_bits(float v) {   // v >= 0, not NaN; the max as FP64 bits
  const float m = __uint_as_float(__reduce_max_sync(FULL_MASK, __float_as_uint(v)));
  return (unsigned long long)__double_as_longlong((double)m);
}
__device__ __forceinline__ unsigned long long warp_max_bits(double v) {
  unsigned long long b = (unsigned long long)__double_as_longlong(v);
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) {
    const unsigned long long o = __shfl_xor_sync(FULL_MASK, b, d);
    b = o > b ? o : b;
  }
  return b;
}

// Sums of NV values over a 256-thread CTA, valid in lane 0 of warp c for value c: warp c adds the eight rows of
// its value, then its 32 lanes (13 warp instructions a value instead of 40).
template <int NV>
__device__ __forceinline__ double cta_sums(const double (&v)[NV], double (&buf)[NV][RED_THREADS]) {
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
  for (int c = 0; c < NV; ++c) buf[c][threadIdx.x] = v[c];
  __syncthreads();
  double s = 0.0;
  if (w < NV) {
    double a[RED_THREADS / 32];
#pragma unroll
    for (int i = 0; i < RED_THREADS / 32; ++i) a[i] = buf[w][32 * i + lane];
    s = ((a[0] + a[1]) + (a[2] + a[3])) + ((a[4] + a[5]) + (a[6] + a[7]));
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) s += __shfl_xor_sync(FULL_MASK, s, d);
  }
  return s;
}

// Per point, the sums over its virtual points of V_v and w'_v: C and w of the physical point (Eq. 15).  A warp
// takes 32 consecutive points; their virtual points are one contiguous range of records, which the warp
// moves through shared memory 32 records at a time with coalesced loads, each lane adding up its own
// point's records in order (no atomics: the sums do not depend on the launch).
template <typename real>
__global__ void __launch_bounds__(256) k_pt_acc(DevProblem P, const real* vp_acc, real* __restrict__ pt_acc) {
  chain_begin();
  __shared__ __align__(16) real stage[8][288];
  const int lane = threadIdx.x & 31;
  real* sm = stage[threadIdx.x >> 5];
  const long long wstride = ((long long)gridDim.x * blockDim.x) >> 5;
  for (long long w = (blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5; w * 32 < P.n; w += wstride) {
    const long long i0 = w * 32;
    const int cnt = (int)(P.n - i0 < 32 ? P.n - i0 : 32);
    const int i = (int)i0 + lane;
    const long long vb = lane < cnt ? P.pt_vp_off[i] : 0, ve = lane < cnt ? P.pt_vp_off[i + 1] : 0;
    const long long r0 = __shfl_sync(FULL_MASK, vb, 0), r1 = __shfl_sync(FULL_MASK, ve, cnt - 1);
    real acc[9];
#pragma unroll
    for (int c = 0; c < 9; ++c) acc[c] = real(0);
    for (long long r = r0; r < r1; r += 32) {   // records [r, r + nr) of the warp's range
      const int nr = (int)(r1 - r < 32 ? r1 - r : 32);
      const real* blk = vp_acc + 9 * r;
      for (int k = lane; k < 9 * nr; k += 32) sm[k] = blk[k];
      __syncwarp();
      const long long ub = vb > r ? vb : r, ue = ve < r + nr ? ve : r + nr;
      for (long long u = ub; u < ue; ++u)
#pragma unroll
        for (int c = 0; c < 9; ++c) acc[c] += sm[9 * (u - r) + c];
      __syncwarp();
    }
    warp_store_rec(pt_acc, i0, cnt, sm, lane, acc);
  }
}

// Warp chunks of 32 virtual points (the first ceil(nv / 32)), then of 32 points; records move through shared
// memory as whole 16-byte vectors.  Virtual point v: L_v^-1 of V'_v = V_v + lambda diag(V_v) and
// y_v = V'_v^-1 w'_v, where on a corrected step w'_v = diag(V_v) dbar_i, dbar_i = w_i / diag(C_i) (Sec. 4.3).
// Point i: C_i^-1 of C_i + lambda diag(C_i), the uncorrected w_i, and max |w| for the stop test.  C_i and w_i
// come from k_pt_acc, or from pt_sums (FP64, summed over every process's virtual points) when the iteration
// is sharded.
template <typename real>
__global__ void __launch_bounds__(256) k_vp_finalize(DevProblem P, Scratch<real> W, DevState* st,
                                                     const double* pt_sums,
                                                     const long long* __restrict__ counts) {
  chain_begin();
  __shared__ __align__(16) real stage[8][32 * VPI];
  const real lam = (real)st->lambda_used;
  const bool corr = st->corrected != 0;
  const long long nv = counts[0];
  const int lane = threadIdx.x & 31;
  real* sm = stage[threadIdx.x >> 5];
  real gmax = real(0);
  // C_i (6 packed) and w_i (3) of point i, read directly (corrected steps)
  auto point_sums = [&](int i, real (&a)[9]) {
    if (pt_sums) {
#pragma unroll
      for (int c = 0; c < 9; ++c) a[c] = (real)pt_sums[9 * (size_t)i + c];
    } else if (P.pt_vp_off[i] == P.pt_vp_off[i + 1]) {   // no observation
#pragma unroll
      for (int c = 0; c < 9; ++c) a[c] = real(0);
    } else {
#pragma unroll
      for (int c = 0; c < 9; ++c) a[c] = W.pt_acc[9 * (size_t)i + c];
    }
  };
  const long long nvc = (nv + 31) / 32, npc = ((long long)P.n + 31) / 32;
  const long long wstride = ((long long)gridDim.x * blockDim.x) >> 5;
  for (long long ch = (blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5; ch < nvc + npc; ch += wstride) {
    real a[9], o[9];
#pragma unroll
    for (int c = 0; c < 9; ++c) a[c] = o[c] = real(0);
    if (ch < nvc) {
      const long long v0 = ch * 32, v = v0 + lane;
      const int cnt = (int)(nv - v0 < 32 ? nv - v0 : 32);
      warp_load_rec9(W.vp_acc, v0, cnt, sm, lane, a);
      const bool other = pt_sums && a[0] == real(0) && a[3] == real(0) && a[5] == real(0);   // another process's
      real X[3] = {0, 0, 0};
      if (lane < cnt) load_point_w(P, P.vp_point[v], X);
      if (lane < cnt && !other) {
        real V[6] = {a[0], a[1], a[2], a[3], a[4], a[5]}, wv[3] = {a[6], a[7], a[8]};
        if (corr) {
          real s[9];
          point_sums(P.vp_point[v], s);
          wv[0] = V[0] * (s[6] / s[0]);
          wv[1] = V[3] * (s[7] / s[3]);
          wv[2] = V[5] * (s[8] / s[5]);
        }
        V[0] += lam * V[0];
        V[3] += lam * V[3];
        V[5] += lam * V[5];
        real Li[6], y[3];
        chol3_inv(V, Li);
        chol3_apply(Li, wv, y);
#pragma unroll
        for (int c = 0; c < 6; ++c) o[c] = Li[c];
#pragma unroll
        for (int c = 0; c < 3; ++c) o[6 + c] = y[c];
      }
      const real rec[VPI] = {o[0], o[1], o[2], o[3], o[4], o[5], X[0], X[1], X[2], o[6], o[7], o[8]};
      warp_store_rec(W.vp_info, v0, cnt, sm, lane, rec);
    } else {
      // physical point: C + lambda diag(C), its inverse, uncorrected w
      const long long i0 = (ch - nvc) * 32;
      const int i = (int)(i0 + lane);
      const int cnt = (int)(P.n - i0 < 32 ? P.n - i0 : 32);
      if (pt_sums) {
        if (lane < cnt) point_sums(i, a);
      } else {
        warp_load_rec9(W.pt_acc, i0, cnt, sm, lane, a);
        if (lane < cnt && P.pt_vp_off[i] == P.pt_vp_off[i + 1]) {   // no observation
#pragma unroll
          for (int c = 0; c < 9; ++c) a[c] = real(0);
        }
      }
      if (lane < cnt) {
        const real Cd[6] = {a[0] * (1 + lam), a[1], a[2], a[3] * (1 + lam), a[4], a[5] * (1 + lam)};
        real Li[6];
        chol3_inv(Cd, Li);
        // C^-1 = L^-T L^-1 (symmetric packed 00 01 02 11 12 22)
        o[0] = Li[0] * Li[0] + Li[1] * Li[1] + Li[3] * Li[3];
        o[1] = Li[1] * Li[2] + Li[3] * Li[4];
        o[2] = Li[3] * Li[5];
        o[3] = Li[2] * Li[2] + Li[4] * Li[4];
        o[4] = Li[4] * Li[5];
        o[5] = Li[5] * Li[5];
        o[6] = a[6];
        o[7] = a[7];
        o[8] = a[8];
        gmax = fmax(gmax, fmax(fabs(a[6]), fmax(fabs(a[7]), fabs(a[8]))));
      }
      warp_store_rec(W.pt_info, i0, cnt, sm, lane, o);
    }
  }
  __shared__ unsigned long long wmax[8];
  const unsigned long long wm = warp_max_bits(gmax);
  if (lane == 0) wmax[threadIdx.x >> 5] = wm;
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned long long b = 0;
#pragma unroll
    for (int i = 0; i < 8; ++i) b = wmax[i] > b ? wmax[i] : b;
    atomicMax(&st->grad_max_bits, b);
  }
}

template <typename real>
void launch_vp_finalize(const DevProblem& P, Scratch<real> W, DevState* st, const long long* counts,
                        cudaStream_t stream, const double* pt_sums) {
  // grids sized by the largest nv (q); the kernels read nv from the device counter
  const long long nmax = (long long)P.q + P.n + 31;
  const long long cap = 8LL * num_sms();
  if (!pt_sums)
    launch_after(chained(P), k_pt_acc<real>, (int)std::min<long long>(((long long)P.n + 255) / 256, cap), 256, stream,
                 P, W.vp_acc, W.pt_acc);
  const int grid = (int)std::min<long long>((nmax + 255) / 256, cap);
  if (pt_sums)   // after an exchange, not a kernel
    k_vp_finalize<real><<<grid, 256, 0, stream>>>(P, W, st, pt_sums, counts);
  else
    launch_after(chained(P), k_vp_finalize<real>, grid, 256, stream, P, W, st, pt_sums, counts);
}

template <typename real>
__global__ void k_pt_sums(DevProblem P, const real* __restrict__ vp_acc, double* __restrict__ out) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < P.n; i += gridDim.x * blockDim.x) {
    double s[9] = {0, 0, 0, 0, 0, 0, 0, 0, 0};
    for (int v = P.pt_vp_off[i]; v < P.pt_vp_off[i + 1]; ++v)
#pragma unroll
      for (int c = 0; c < 9; ++c) s[c] += (double)vp_acc[9 * (size_t)v + c];
#pragma unroll
    for (int c = 0; c < 9; ++c) out[9 * (size_t)i + c] = s[c];
  }
}

template <typename real>
void launch_pt_sums(const DevProblem& P, Scratch<real> W, double* out, cudaStream_t stream) {
  k_pt_sums<real><<<std::min((P.n + 255) / 256, 4096), 256, 0, stream>>>(P, W.vp_acc, out);
}

template <typename real>
__global__ void k_step_rows(int m, const real* __restrict__ ctab, const double* __restrict__ dc, real* __restrict__ edc) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < 9 * (int64_t)m; i += (int64_t)gridDim.x * blockDim.x) {
    const int j = (int)(i / 9), c = (int)(i - 9 * (int64_t)j);
    edc[(size_t)VPI * j + c] = step_entry(jl_ptr(ctab, m, j), dc + 9 * (size_t)j, c);
  }
}

template <typename real>
void launch_step_rows(const DevProblem& P, const double* dc, real* edc, cudaStream_t stream) {
  const real* ctab;
  if constexpr (sizeof(real) == 4) ctab = P.ctab_f; else ctab = P.ctab_d;
  k_step_rows<real><<<(int)std::min<int64_t>((9 * (int64_t)P.m + 255) / 256, 4096), 256, 0, stream>>>(P.m, ctab, dc, edc);
}

__global__ void k_failed_io(DevState* st, double* x, int to_double) {
  if (threadIdx.x == 0 && blockIdx.x == 0) {
    if (to_double)
      *x = (double)st->failed;
    else
      st->failed = (int)(*x + 0.5);
  }
}

void launch_failed_io(DevState* st, double* x, int to_double, cudaStream_t stream) {
  k_failed_io<<<1, 32, 0, stream>>>(st, x, to_double);
}

// ------------------------------------------------------------------------------------------------------
// S' build (Eq. 10/13), in two passes.  With V' = L L^T the Cholesky factor of a virtual point's damped
// block and, for each of its observations, Pm_o = L^-1 Jp,o^T (3x2), the Schur term of two observations is
// E' C'^-1 E'^T = Jc,a^T (Pm_a^T Pm_b) Jc,b with a 2x2 middle, so
//   off-diagonal camera blocks   S(a, b) = - sum_v Jc,a^T (Pm_a^T Pm_b) Jc,b          (k_pair_build)
//   diagonal camera block        S(a, a) = sum_o [Jc^T (I - Pm_o^T Pm_o) Jc + lambda diag(Jc^T Jc)]  (k_cam_pass)
//   right-hand side              b(a)    = - sum_o Jc^T (f_o + Jp,o y_v),  y_v = V'^-1 w'_v
//   camera gradient              v(a)    = - sum_o Jc^T f_o
// For a virtual point with one observation, I - Pm^T Pm = I - Jp V'^-1 Jp^T cancels by a
// factor ~ lambda; it is evaluated in the equivalent Woodbury form (I + Jp Lambda^-1 Jp^T)^-1 with
// Lambda = lambda diag(Jp^T Jp), and without correction b(a) gets -Jc^T (I + Jp Lambda^-1 Jp^T)^-1 f_o.
//
// k_cam_pass: one warp per 32 observations of one camera (each camera's observation list is padded to
// whole warps on the host, single-observation virtual points first so that warps mostly run one branch).
// Every thread forms the 45 + 9 + 9 terms of its observation; the warp sums them in the working precision
// with a transposed reduction (62 shuffles leave lane L with the sums of terms L and 32 + L; a tree sum of
// 32 terms, error <= 5 ulp of the sum of magnitudes) and adds them atomically into the FP64 S', b' and v
// (zeroed before the launch): FP32 terms, FP64 accumulation across warps.  The per-observation arithmetic
// stays off the FP64 pipe, which on this GPU runs at 1/64 of the FP32 rate.  With stored pair rows it also
// stores (Pm_o, the tilde rows of Jc,o) of every observation of a multi-observation virtual point.
// Both passes evaluate the same rows (stba_camtab.cuh; in FP32 with every operation rounded on its own): the
// diagonal and off-diagonal blocks of a virtual point come from bitwise the same Jt and J_p whether they are
// stored or recomputed, and the FP32 S' does not change with the compiler's choice of fused multiply-adds.  The
// constant factor Jl of the three rotation columns is rounded in per observation here and once per block in the pair
// pass; with it per observation in both, the solution of S' x = b' is as far from FP64 as this way (lambda 1e-5 to
// 0.05, ten systems of each of five kinds: medians within 7 %), and S' and b' themselves are closer to FP64 than
// from rows that evaluate Rodrigues' formula (off-diagonal blocks of 1000 photos 3.9e-9 of the unit diagonal, 5.5e-9).
constexpr int ROWREC = 24;   // reals per stored observation: Pm (6), tilde rows of J_c (18)

// On return lane L holds the sum over the warp's lanes of v[L].  Each halving step keeps one half of the
// values (lanes whose bit s is set keep the upper half) and adds the partner's copy of it.
template <typename real>
__device__ __forceinline__ real warp_transpose_sum32(real (&v)[32]) {
  const int lane = threadIdx.x & 31;
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
  return v[0];
}

// Pm = L^-1 Jp^T (3 x 2) of one observation, with every product and sum rounded by explicit fma / mul intrinsics,
// so that the camera pass and the pair pass form bitwise the same values from the same inputs (the S' of a
// virtual point then stays consistent between its diagonal and off-diagonal camera blocks).
__device__ __forceinline__ float fma_rn(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double fma_rn(double a, double b, double c) { return __fma_rn(a, b, c); }
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }

template <typename real>
__device__ __forceinline__ void pm_of_obs(const real* Li, const real (&Jp)[2][3], real (&Pm)[3][2]) {
#pragma unroll
  for (int t = 0; t < 2; ++t) {
    Pm[0][t] = mul_rn(Li[0], Jp[t][0]);
    Pm[1][t] = fma_rn(Li[2], Jp[t][1], mul_rn(Li[1], Jp[t][0]));
    Pm[2][t] = fma_rn(Li[5], Jp[t][2], fma_rn(Li[4], Jp[t][1], mul_rn(Li[3], Jp[t][0])));
  }
}

template <typename real>
__global__ void __launch_bounds__(256, sizeof(real) == 4 ? 4 : 3) k_cam_pass(DevProblem P, Scratch<real> W, CamSlots CS,
                                                                             real* rowbuf, const DevState* st) {
  const int gw = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (gw >= CS.nwarps) return;   // uniform per warp
  const int lane = threadIdx.x & 31;
  const int j = CS.warp_cam[gw];
  if (P.sharded && !P.cluster_owned[P.cam_cluster[j]]) return;   // another process's cluster (uniform per warp)
  const int o = CS.slots[32 * (size_t)gw + lane];
  const real lam = (real)st->lambda_used;
  const bool corr = st->corrected != 0;
  real Jc[2][9], N00 = 0, N01 = 0, N11 = 0, br[2] = {0, 0}, r[2] = {0, 0};
#pragma unroll
  for (int c = 0; c < 9; ++c) Jc[0][c] = Jc[1][c] = 0;
  if (o >= 0) {
    const CamRow<real> C = load_camrow<real>(P, j);
    // virtual point of the slot (its record holds the point), stored in slot order with the camera lists
    const int pvs = CS.pv[32 * (size_t)gw + lane].y;
    const int v = pvs & INT_MAX;
    const bool single = pvs < 0;
    real vi[VPI], Jp[2][3], Jl[9];
    load_vec16<VPI>(W.vp_info + (size_t)VPI * v, vi);
    const real X[3] = {vi[VPI_X], vi[VPI_X + 1], vi[VPI_X + 2]};
    load_jl(P, j, Jl);
    proj_rows<real, true>(C, X, Jc, Jp);   // tilde rows
    r[0] = res_ptr<real>(P)[2 * (size_t)o];
    r[1] = res_ptr<real>(P)[2 * (size_t)o + 1];
    scale_rows(row_weight(P, r[0], r[1]), r, Jc, Jp);
    // Both cases reduce to Jc^T N Jc with a 2x2 N:
    //   single observation  N = (I + Jp Lambda^-1 Jp^T)^-1                 (Woodbury, no cancellation)
    //   several             N = I - Jp V'^-1 Jp^T = I - P^T P, P = L^-1 Jp^T  (V' = L L^T)
    if (single) {
      real il[3];
#pragma unroll
      for (int s = 0; s < 3; ++s) il[s] = real(1) / (lam * (Jp[0][s] * Jp[0][s] + Jp[1][s] * Jp[1][s]));
      real K00 = 0, K01 = 0, K11 = 0;
#pragma unroll
      for (int s = 0; s < 3; ++s) {
        K00 += Jp[0][s] * Jp[0][s] * il[s];
        K01 += Jp[0][s] * Jp[1][s] * il[s];
        K11 += Jp[1][s] * Jp[1][s] * il[s];
      }
      const real idet = real(1) / ((real(1) + K00) * (real(1) + K11) - K01 * K01);
      N00 = (real(1) + K11) * idet;
      N01 = -K01 * idet;
      N11 = (real(1) + K00) * idet;
      if (corr) {
        br[0] = r[0] + Jp[0][0] * vi[VPI_Y] + Jp[0][1] * vi[VPI_Y + 1] + Jp[0][2] * vi[VPI_Y + 2];
        br[1] = r[1] + Jp[1][0] * vi[VPI_Y] + Jp[1][1] * vi[VPI_Y + 1] + Jp[1][2] * vi[VPI_Y + 2];
      } else {
        br[0] = N00 * r[0] + N01 * r[1];
        br[1] = N01 * r[0] + N11 * r[1];
      }
    } else {
      real Pm[3][2];
      pm_of_obs<real>(vi, Jp, Pm);
      N00 = real(1) - (Pm[0][0] * Pm[0][0] + Pm[1][0] * Pm[1][0] + Pm[2][0] * Pm[2][0]);
      N01 = -(Pm[0][0] * Pm[0][1] + Pm[1][0] * Pm[1][1] + Pm[2][0] * Pm[2][1]);
      N11 = real(1) - (Pm[0][1] * Pm[0][1] + Pm[1][1] * Pm[1][1] + Pm[2][1] * Pm[2][1]);
      if (!P.pair_recompute) {   // the pair pass's rows, with 16-byte stores, indexed like the camera graph's pairs
        real v24[ROWREC];
#pragma unroll
        for (int t = 0; t < 6; ++t) v24[t] = Pm[t >> 1][t & 1];
#pragma unroll
        for (int c = 0; c < 9; ++c) {
          v24[6 + 2 * c] = Jc[0][c];
          v24[7 + 2 * c] = Jc[1][c];
        }
        real* dst = rowbuf + (size_t)ROWREC * P.obs_base[o];
        if constexpr (sizeof(real) == 4) {
#pragma unroll
          for (int k = 0; k < ROWREC / 4; ++k)
            reinterpret_cast<float4*>(dst)[k] = make_float4(v24[4 * k], v24[4 * k + 1], v24[4 * k + 2], v24[4 * k + 3]);
        } else {
#pragma unroll
          for (int k = 0; k < ROWREC / 2; ++k) reinterpret_cast<double2*>(dst)[k] = make_double2(v24[2 * k], v24[2 * k + 1]);
        }
      }
      br[0] = r[0] + Jp[0][0] * vi[VPI_Y] + Jp[0][1] * vi[VPI_Y + 1] + Jp[0][2] * vi[VPI_Y + 2];
      br[1] = r[1] + Jp[1][0] * vi[VPI_Y] + Jp[1][1] * vi[VPI_Y + 1] + Jp[1][2] * vi[VPI_Y + 2];
    }
    apply_jl<real>(Jl, Jc);
  }
  // terms: 0..44 diagonal block (packed lower, row-major), 45..53 b', 54..62 v, 63 unused
  real NJ[2][9];
#pragma unroll
  for (int c = 0; c < 9; ++c) {
    NJ[0][c] = N00 * Jc[0][c] + N01 * Jc[1][c];
    NJ[1][c] = N01 * Jc[0][c] + N11 * Jc[1][c];
  }
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
          real d = Jc[0][i] * NJ[0][jj] + Jc[1][i] * NJ[1][jj];
          if (i == jj) d += lam * (Jc[0][i] * Jc[0][i] + Jc[1][i] * Jc[1][i]);
          v[t - 32 * half] = d;
        }
      }
    if (half == 1) {
#pragma unroll
      for (int i = 0; i < 9; ++i) {
        v[45 - 32 + i] = -(Jc[0][i] * br[0] + Jc[1][i] * br[1]);
        v[54 - 32 + i] = -(Jc[0][i] * r[0] + Jc[1][i] * r[1]);
      }
      v[31] = real(0);
    }
    sums[half] = warp_transpose_sum32(v);
  }
  const int k = P.cam_cluster[j], lc = P.cam_local[j];
  const int np = P.cluster_np[k];
#pragma unroll
  for (int half = 0; half < 2; ++half) {
    const int e = lane + 32 * half;
    const double x = (double)sums[half];
    if (e < 45) {
      int row = 0;
      while ((row + 1) * (row + 2) / 2 <= e) ++row;
      const int col = e - row * (row + 1) / 2;
      atomicAdd(W.S + P.S_off[k] + (size_t)(9 * lc + row) * np + 9 * lc + col, x);
    } else if (e < 54) {
      atomicAdd(W.b + P.v_off[k] + 9 * lc + (e - 45), x);
    } else if (e < 63) {
      atomicAdd(W.vgrad + 9 * (size_t)j + (e - 54), sums[half]);
    }
  }
}

// k_pair_build: the off-diagonal blocks S'_k(la, lb) = -sum over the points seen by both cameras x > y of
// one cluster of Jc,x^T (Pm_x^T Pm_y) Jc,y (Eq. 10, 13).  The observation pairs of the camera graph are listed
// once, at create, by edge (x, y) and cut into chunks (pair_chunk); under a cluster assignment an edge
// contributes exactly when both cameras are in one cluster (its two observations of a point are then in
// one virtual point), and a chunk adds to one block only.  The re-ordering of an assignment lists the
// chunks whose edge lies inside a cluster; the warps of a fixed grid take them one by one from that list.  A warp
// works on pieces of PB_CH pairs: lane (side, j) forms the rows of its pair's observation by camera x (side 0) or y
// (side 1) from the camera's table, the point and L_v^-1 (both lanes of a pair share them); the y lane takes Pm_x by
// shuffle and forms M = Pm_x^T Pm_y (2x2) and M Jt_y (2x9).  The rows go to shared memory, and 27 lanes accumulate: lane
// (g, rb, cb) takes every third pair (slot g) and the 3 x 3 sub-block (rb, cb), in FP32 as packed pairs of FMAs
// over the rank index.  The three slots are summed by two shuffles, the block is multiplied by the cameras' Jl
// (J_c = Jt E) and written once per chunk to the FP64 S'_k: stored when the chunk is its edge's only one (the
// edge's block has no other writer), else added atomically.
// Bound by the L1 / shared-memory pipe (ncu: 85 % of its wavefronts): per 16 pairs about 65 wavefronts of row reads,
// 26 of row writes, 80 of the gathers of the 48-byte virtual-point records.  Hence rank-2 rows (3x9 blocks
// G = L^-1 Jp^T Jc of both sides move half as many words again), 16-byte records and loads, 24 warps per SM
// (80 registers; 32 warps spill: 150 us against 135 us for 2.9M pairs).  S' build stage, before -> now:
// 1000 cameras, 2.9M pairs 316 -> 177 us; 2000 sequential cameras, 10.5M pairs 913 -> 483; 6000 cameras, 12M
// pairs 1802 -> 774; FP64, 300 cameras, 0.5M pairs 2702 -> 574 (stored rows: bound by the FP64 pipe).
constexpr int PB_WARPS = 8;
constexpr int PB_CH = 16;   // pairs per piece: one per lane and side
template <typename real> constexpr int pb_ctas() { return sizeof(real) == 4 ? 3 : 2; }   // resident CTAs per SM

// Shared-memory rows of a piece: per pair and side three groups (camera-parameter triples) of 3 columns x 2 ranks,
// 16-byte aligned; the pair stride spreads the 16-byte stores of 8 consecutive lanes over all banks.
template <typename real> struct PairRows {
  static constexpr int GROUP = sizeof(real) == 4 ? 8 : 6, SIDE = 3 * GROUP, PAIR = sizeof(real) == 4 ? 52 : 50;
  static constexpr size_t bytes = sizeof(real) * (size_t)PB_WARPS * PB_CH * PAIR;
};

// 3 columns x 2 ranks of one group
template <typename real>
__device__ __forceinline__ void store_group(real* dst, const real (&v)[6]) {
  if constexpr (sizeof(real) == 4) {
    *reinterpret_cast<float4*>(dst) = make_float4(v[0], v[1], v[2], v[3]);
    *reinterpret_cast<float2*>(dst + 4) = make_float2(v[4], v[5]);
  } else {
#pragma unroll
    for (int k = 0; k < 3; ++k) *reinterpret_cast<double2*>(dst + 2 * k) = make_double2(v[2 * k], v[2 * k + 1]);
  }
}
template <typename real>
__device__ __forceinline__ void load_group(const real* src, real (&v)[6]) {
  if constexpr (sizeof(real) == 4) {
    const float4 a = *reinterpret_cast<const float4*>(src);
    const float2 b = *reinterpret_cast<const float2*>(src + 4);
    v[0] = a.x;
    v[1] = a.y;
    v[2] = a.z;
    v[3] = a.w;
    v[4] = b.x;
    v[5] = b.y;
  } else {
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const double2 t = *reinterpret_cast<const double2*>(src + 2 * k);
      v[2 * k] = t.x;
      v[2 * k + 1] = t.y;
    }
  }
}

// Accumulator of a 2-term product sum: FP32 as one packed pair of FMAs (the two ranks side by side, added at the
// end), FP64 as two FMAs.
template <typename real> struct Acc2;
template <> struct Acc2<float> {
  unsigned long long v;
  __device__ __forceinline__ void zero() { v = 0ull; }
  __device__ __forceinline__ void add(float a0, float a1, float b0, float b1) {
    asm("{\n.reg .b64 a, b;\nmov.b64 a, {%1, %2};\nmov.b64 b, {%3, %4};\nfma.rn.f32x2 %0, a, b, %0;\n}"
        : "+l"(v)
        : "f"(a0), "f"(a1), "f"(b0), "f"(b1));
  }
  __device__ __forceinline__ float sum() const {
    float lo, hi;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
    return lo + hi;
  }
};
template <> struct Acc2<double> {
  double v;
  __device__ __forceinline__ void zero() { v = 0.0; }
  __device__ __forceinline__ void add(double a0, double a1, double b0, double b1) { v = fma(a1, b1, fma(a0, b0, v)); }
  __device__ __forceinline__ double sum() const { return v; }
};

template <typename real, bool RECOMPUTE>
__global__ void __launch_bounds__(32 * PB_WARPS, pb_ctas<real>())
    k_pair_build(DevProblem P, Scratch<real> W, PairChunks B, const real* __restrict__ rowbuf, DevState* st) {
  using PR = PairRows<real>;
  extern __shared__ __align__(16) unsigned char pb_smem[];
  const int wib = threadIdx.x >> 5, lane = threadIdx.x & 31;
  real* stage = reinterpret_cast<real*>(pb_smem) + (size_t)wib * PB_CH * PR::PAIR;
  const long long nactive = *B.nactive;
  // chunks are handed out by a counter (zeroed with the iteration): their sizes vary, and a fixed stride leaves the
  // most loaded warp half as much again as the average
  auto take = [&]() {
    unsigned w = 0;
    if (lane == 0) w = atomicAdd(&st->pair_next, 1u);
    return (long long)__shfl_sync(FULL_MASK, w, 0);
  };
  const long long w0 = take();
  if (w0 >= nactive) return;   // uniform per warp
  // lanes 0..26: pair slot g = lane / 9 of every three, and the 3 x 3 sub-block (rb, cb) of the 9 x 9 block
  const int g = lane / 9, sub = lane - 9 * (lane / 9), rb = sub / 3, cb = sub - 3 * (sub / 3);
  const int j = lane % PB_CH, side = lane / PB_CH;
  int4 ch = B.chunks[B.active[w0]];
  long long wn = take();   // the warp's next chunk
  int4 chn = B.chunks[B.active[min(wn, nactive - 1)]];
  int c0 = 0;
  // the pair of this lane in the piece at (chunk, first), and the virtual point of its observations
  auto pair_of = [&](const int4& chunk, int first) {
    return B.pairs[chunk.z + min(first + j, (chunk.w & PAIR_COUNT_MASK) - 1)];
  };
  int2 pr = pair_of(ch, 0);
  int vp = RECOMPUTE ? P.base_vp[pr.x] : 0;
  Acc2<real> acc[3][3];
#pragma unroll
  for (int x = 0; x < 3; ++x)
#pragma unroll
    for (int y = 0; y < 3; ++y) acc[x][y].zero();
  for (;;) {
    // the next piece: the rest of this chunk, else the warp's next chunk
    const int count = ch.w & PAIR_COUNT_MASK;
    int4 nch = ch;
    int n0 = c0 + PB_CH;
    bool more = true;
    if (n0 >= count) {
      nch = chn;
      n0 = 0;
      more = wn < nactive;
    }
    // rows of this lane's observation (a lane past the chunk's end repeats its last pair; it is not accumulated)
    real Pm[3][2], Jt[2][9];
    if constexpr (RECOMPUTE) {
      const CamRow<real> C = load_camrow<real>(P, side ? ch.y : ch.x);
      real vi[VPI], Jp[2][3];   // L_v^-1 and the point
      load_vec16<VPI>(W.vp_info + (size_t)VPI * vp, vi);
      const real X[3] = {vi[VPI_X], vi[VPI_X + 1], vi[VPI_X + 2]};
      proj_rows<real, true>(C, X, Jt, Jp);
      if (P.huber_a > 0.0) {
        const size_t pos = (size_t)P.base_pos[side ? pr.y : pr.x];
        real r[2] = {res_ptr<real>(P)[2 * pos], res_ptr<real>(P)[2 * pos + 1]};
        scale_rows(row_weight(P, r[0], r[1]), r, Jt, Jp);
      }
      pm_of_obs<real>(vi, Jp, Pm);
    } else {
      real v24[ROWREC];
      load_vec16<ROWREC>(rowbuf + (size_t)ROWREC * (side ? pr.y : pr.x), v24);
#pragma unroll
      for (int t = 0; t < 6; ++t) Pm[t >> 1][t & 1] = v24[t];
#pragma unroll
      for (int c = 0; c < 9; ++c) {
        Jt[0][c] = v24[6 + 2 * c];
        Jt[1][c] = v24[7 + 2 * c];
      }
    }
    // the next piece's pairs (their virtual points follow below, once these have arrived)
    int2 prn = pr;
    if (more) prn = pair_of(nch, n0);
    // y lanes: rows M Jt_y with M = Pm_x^T Pm_y
    real M[2][2] = {{0, 0}, {0, 0}};
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const real a0 = __shfl_sync(FULL_MASK, Pm[k][0], j), a1 = __shfl_sync(FULL_MASK, Pm[k][1], j);
      M[0][0] += a0 * Pm[k][0];
      M[0][1] += a0 * Pm[k][1];
      M[1][0] += a1 * Pm[k][0];
      M[1][1] += a1 * Pm[k][1];
    }
    real* dst = stage + (size_t)j * PR::PAIR + side * PR::SIDE;
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      real v6[6];
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const real u0 = Jt[0][3 * b + c], u1 = Jt[1][3 * b + c];
        v6[2 * c] = side ? M[0][0] * u0 + M[0][1] * u1 : u0;
        v6[2 * c + 1] = side ? M[1][0] * u0 + M[1][1] * u1 : u1;
      }
      store_group<real>(dst + b * PR::GROUP, v6);
    }
    __syncwarp();
    if (RECOMPUTE && more) vp = P.base_vp[prn.x];
    if (lane < 27) {
      const int cn = min(PB_CH, count - c0);
      for (int jj = g; jj < cn; jj += 3) {   // pair slot g of every three
        real a[6], b[6];
        load_group<real>(stage + (size_t)jj * PR::PAIR + rb * PR::GROUP, a);
        load_group<real>(stage + (size_t)jj * PR::PAIR + PR::SIDE + cb * PR::GROUP, b);
#pragma unroll
        for (int x = 0; x < 3; ++x)
#pragma unroll
          for (int y = 0; y < 3; ++y) acc[x][y].add(a[2 * x], a[2 * x + 1], b[2 * y], b[2 * y + 1]);
      }
    }
    __syncwarp();   // every lane is done with the rows before they are overwritten
    if (c0 + PB_CH >= count) {   // the chunk is complete: sum the three pair slots, write the block
      real s[3][3];
#pragma unroll
      for (int x = 0; x < 3; ++x)
#pragma unroll
        for (int y = 0; y < 3; ++y) {
          // lane L < 9 adds slots 1 and 2 from lanes L + 9 and L + 18 (source lanes wrap mod 32 for the rest)
          const real v = acc[x][y].sum();
          s[x][y] = v + __shfl_sync(FULL_MASK, v, lane + 9) + __shfl_sync(FULL_MASK, v, lane + 18);
          acc[x][y].zero();
        }
      if (lane < 9) {
        // the rotation rows and columns: J_c = Jt E
        real Jl[9], t[3][3];
        if (rb == 0) {
          load_jl(P, ch.x, Jl);
#pragma unroll
          for (int x = 0; x < 3; ++x)
#pragma unroll
            for (int y = 0; y < 3; ++y) t[x][y] = Jl[x] * s[0][y] + Jl[3 + x] * s[1][y] + Jl[6 + x] * s[2][y];
#pragma unroll
          for (int x = 0; x < 3; ++x)
#pragma unroll
            for (int y = 0; y < 3; ++y) s[x][y] = t[x][y];
        }
        if (cb == 0) {
          load_jl(P, ch.y, Jl);
#pragma unroll
          for (int x = 0; x < 3; ++x)
#pragma unroll
            for (int y = 0; y < 3; ++y) t[x][y] = s[x][0] * Jl[y] + s[x][1] * Jl[3 + y] + s[x][2] * Jl[6 + y];
#pragma unroll
          for (int x = 0; x < 3; ++x)
#pragma unroll
            for (int y = 0; y < 3; ++y) s[x][y] = t[x][y];
        }
#pragma unroll
        for (int x = 0; x < 3; ++x)
#pragma unroll
          for (int y = 0; y < 3; ++y) stage[9 * (3 * rb + x) + 3 * cb + y] = s[x][y];
      }
      __syncwarp();
      const int k = P.cam_cluster[ch.x];
      const int la = P.cam_local[ch.x], lb = P.cam_local[ch.y];   // la > lb: local order follows camera order
      const int np = P.cluster_np[k];
      double* dstS = W.S + P.S_off[k] + (size_t)(9 * la) * np + 9 * lb;
      if (lane < 27) {   // three rows of the block per instruction
#pragma unroll
        for (int t = 0; t < 3; ++t) {
          const int row = 3 * t + g;
          double* d = dstS + (size_t)row * np + sub;
          const double v = -(double)stage[9 * row + sub];
          if (ch.w & PAIR_WHOLE_EDGE)
            *d = v;
          else
            atomicAdd(d, v);
        }
      }
      __syncwarp();   // the rows are overwritten next
      if (!more) break;
      wn = take();
      chn = B.chunks[B.active[min(wn, nactive - 1)]];
    }
    ch = nch;
    c0 = n0;
    pr = prn;
  }
}

template <typename real>
void launch_rcs_build(const DevProblem& P, Scratch<real> W, CamSlots CS, PairChunks B, real* rowbuf, DevState* st,
                      cudaStream_t stream, cudaStream_t side, cudaEvent_t fork, cudaEvent_t join) {
  const bool pairs = B.nchunks > 0 && P.l < P.m;
  // a pair pass that recomputes its rows depends on nothing the camera pass writes (they add to different
  // blocks of S'), so with a second stream the two run side by side
  const bool beside = pairs && P.pair_recompute && side != nullptr;
  if (beside) {
    cudaEventRecord(fork, stream);
    cudaStreamWaitEvent(side, fork, 0);
  }
  cudaStream_t ps = beside ? side : stream;
  k_cam_pass<real><<<(CS.nwarps + 7) / 8, 256, 0, stream>>>(P, W, CS, rowbuf, st);
  if (pairs) {   // a fixed grid takes the chunks inside clusters
    const int grid = std::min((B.nchunks + PB_WARPS - 1) / PB_WARPS, pb_ctas<real>() * num_sms());
    if (P.pair_recompute)
      k_pair_build<real, true><<<grid, 32 * PB_WARPS, PairRows<real>::bytes, ps>>>(P, W, B, rowbuf, st);
    else
      k_pair_build<real, false><<<grid, 32 * PB_WARPS, PairRows<real>::bytes, ps>>>(P, W, B, rowbuf, st);
  }
  if (beside) {
    cudaEventRecord(join, side);
    cudaStreamWaitEvent(stream, join, 0);
  }
}

// ------------------------------------------------------------------------------------------------------
// Double-float numbers: a value is an unevaluated sum hi + lo of two floats.
__device__ __forceinline__ float2 df_two_sum(float a, float b) {
  const float s = a + b;
  const float bb = s - a;
  return make_float2(s, (a - (s - bb)) + (b - bb));
}
__device__ __forceinline__ float2 df_fast_two_sum(float a, float b) {   // |a| >= |b|
  const float s = a + b;
  return make_float2(s, b - (s - a));
}
__device__ __forceinline__ float2 df_add(float2 x, float2 y) {
  const float2 s = df_two_sum(x.x, y.x);
  return df_fast_two_sum(s.x, s.y + (x.y + y.y));
}
__device__ __forceinline__ float2 df_sub(float2 x, float2 y) { return df_add(x, make_float2(-y.x, -y.y)); }
__device__ __forceinline__ float2 df_mul(float2 x, float2 y) {
  const float p = x.x * y.x;
  const float e = fmaf(x.x, y.y, fmaf(x.y, y.x, fmaf(x.x, y.x, -p)));
  return df_fast_two_sum(p, e);
}
__device__ __forceinline__ float2 df_rcp(float2 y) {   // one Newton correction of the FP32 reciprocal
  const float q = __frcp_rn(y.x);
  const float2 r = df_sub(make_float2(1.f, 0.f), df_mul(make_float2(q, 0.f), y));
  return df_fast_two_sum(q, r.x * q);
}
__device__ __forceinline__ float2 df_split(double d) {
  const float hi = __double2float_rn(d);
  return make_float2(hi, __double2float_rn(d - (double)hi));
}

// ------------------------------------------------------------------------------------------------------
template <typename real>
__global__ void __launch_bounds__(256) k_point_rhs(DevProblem P, const real* edc, real* t_acc) {
  chain_begin();
  const int o = blockIdx.x * blockDim.x + threadIdx.x;
  const int lane = threadIdx.x & 31;
  const bool act = o < P.q;
  int pt = INT_MAX;
  real val[3] = {0, 0, 0};
  if (act) {
    pt = P.obs_pt[o];
    const int cam = P.obs_cam[o];
    const CamRow<real> C = gather_camrow<real>(P, cam);
    real X[3];
    load_point_w(P, pt, X);
    real Jt[2][9], Jp[2][3], d[12];
    gather_vec16<12>(edc + (size_t)VPI * cam, d);   // J_c dc = Jt (E dc)
    proj_rows<real, true>(C, X, Jt, Jp);
    real jd0 = 0, jd1 = 0;
#pragma unroll
    for (int c = 0; c < 9; ++c) {
      jd0 += Jt[0][c] * d[c];
      jd1 += Jt[1][c] * d[c];
    }
    // with a robust loss both Jacobians carry sqrt(rho'): the product carries rho'
    real wgt = real(1);
    if (P.huber_a > 0.0) {
      const real sw = huber_sqrt_weight<real>(P.huber_a, res_ptr<real>(P)[2 * (size_t)o], res_ptr<real>(P)[2 * (size_t)o + 1]);
      wgt = sw * sw;
    }
#pragma unroll
    for (int j = 0; j < 3; ++j) val[j] = wgt * (Jp[0][j] * jd0 + Jp[1][j] * jd1);
  }
  segmented_scan<3>(val, pt, lane);
  segmented_store<3>(val, pt, act, lane, o, P.pt_off, t_acc);
}

// dp = C^-1 (w - t) per point; the same grid also forms the partial sums of the stop tests: |dp|^2, |p|^2,
// |dc|^2, |c|^2 and max |v| (camera gradient), one partial per block at partial[RED_BLOCKS * (1..5) + block].
// With pdf (mixed precision) it also writes the candidate p + dp as double-float numbers for k_cost_df.
// Bound by the FP64 pipe: the sums were four shuffle trees in each of the eight warps (14 us at 1000 photos with
// a separate 8 us kernel for the double-float points; the fused kernel takes 15.6 us).
template <typename real>
__global__ void __launch_bounds__(RED_THREADS) k_point_update(DevProblem P, const real* pt_info, const real* t_acc,
                                                              const double* dc, const real* vgrad, double* dp,
                                                              float2* pdf, double* partial) {
  chain_begin();
  double s_dp = 0.0, s_p = 0.0, s_dc = 0.0, s_c = 0.0;
  real gmax = real(0);   // max |v| in the working precision (exact)
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < P.n; i += gridDim.x * blockDim.x) {
    const real* in = pt_info + 9 * (size_t)i;
    const real* t = t_acc + 3 * (size_t)i;
    const double p[3] = {P.pts[3 * (size_t)i], P.pts[3 * (size_t)i + 1], P.pts[3 * (size_t)i + 2]};
    real g0 = in[6] - t[0], g1 = in[7] - t[1], g2 = in[8] - t[2];
    real d0 = in[0] * g0 + in[1] * g1 + in[2] * g2;
    real d1 = in[1] * g0 + in[3] * g1 + in[4] * g2;
    real d2 = in[2] * g0 + in[4] * g1 + in[5] * g2;
    double* out = dp + 3 * (size_t)i;
    out[0] = d0;
    out[1] = d1;
    out[2] = d2;
    const double e[3] = {(double)d0, (double)d1, (double)d2};
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const double pc = p[c];
      s_dp += e[c] * e[c];
      s_p += pc * pc;
      if constexpr (sizeof(real) == 4) pdf[3 * (size_t)i + c] = df_split(pc + e[c]);
    }
  }
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < 9 * P.m; i += gridDim.x * blockDim.x) {
    const double d = dc[i], c = P.cams[i];
    s_dc += d * d;
    s_c += c * c;
    gmax = fmax(gmax, fabs(vgrad[i]));
  }
  __shared__ double buf[4][RED_THREADS];
  __shared__ unsigned long long wmax[RED_THREADS / 32];
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const unsigned long long wm = warp_max_bits(gmax);
  if (lane == 0) wmax[w] = wm;
  const double v[4] = {s_dp, s_p, s_dc, s_c};
  const double a = cta_sums<4>(v, buf);
  if (lane == 0 && w < 4) partial[(1 + w) * RED_BLOCKS + blockIdx.x] = a;
  if (threadIdx.x == 32 * 4) {
    unsigned long long b = 0;
#pragma unroll
    for (int i = 0; i < RED_THREADS / 32; ++i) b = wmax[i] > b ? wmax[i] : b;
    partial[5 * RED_BLOCKS + blockIdx.x] = __longlong_as_double((long long)b);
  }
}

// ------------------------------------------------------------------------------------------------------
// Residuals in FP64 (both precisions): the cost F(x + dx) and the accept test need them to FP64 accuracy,
// and the stored residuals drive the next linearisation (FP32 projections of pixel coordinates of a few
// hundred px carry ~3e-5 px of rounding, which the conditioning of S' amplifies in the step).
// k_cost_cams: per camera R(w + dw) (Rodrigues in FP64), t + dt and the intrinsics, as 15 FP64 numbers, or in
// mixed precision split into double-float (CAM_DF floats).  A long FP64 chain per camera and 16 cycles a warp
// instruction: one warp a CTA, so that the cameras spread over the SMs (four warps a CTA and the split in a
// kernel of its own: 7.9 + 5.3 us at 1000 cameras; 8.4 us now, beside the point step).
constexpr int CAM_DF = 28;   // floats per camera: R (9 x 2), t (3 x 2), f (2), k1, k2

template <typename real>
__global__ void __launch_bounds__(32) k_cost_cams(int m, const double* __restrict__ cams, const double* __restrict__ dc,
                                                  double* __restrict__ rt, float* __restrict__ cdf) {
  const int j = 32 * blockIdx.x + threadIdx.x;
  if (j >= m) return;
  double c[9];
#pragma unroll
  for (int i = 0; i < 9; ++i) c[i] = cams[9 * (size_t)j + i] + (dc ? dc[9 * (size_t)j + i] : 0.0);
  const double s = c[0] * c[0] + c[1] * c[1] + c[2] * c[2];
  double a, b, da, db;
  rodrigues_coeffs(s, a, b, da, db);
  const double* w = c;
  double o[15];
  o[0] = 1.0 + b * (w[0] * w[0] - s);
  o[1] = -a * w[2] + b * w[0] * w[1];
  o[2] = a * w[1] + b * w[0] * w[2];
  o[3] = a * w[2] + b * w[0] * w[1];
  o[4] = 1.0 + b * (w[1] * w[1] - s);
  o[5] = -a * w[0] + b * w[1] * w[2];
  o[6] = -a * w[1] + b * w[0] * w[2];
  o[7] = a * w[0] + b * w[1] * w[2];
  o[8] = 1.0 + b * (w[2] * w[2] - s);
#pragma unroll
  for (int i = 0; i < 6; ++i) o[9 + i] = c[3 + i];
  if constexpr (sizeof(real) == 4) {
    float4* out = reinterpret_cast<float4*>(cdf + CAM_DF * (size_t)j);
#pragma unroll
    for (int i = 0; i < 6; ++i) {
      const float2 u = df_split(o[2 * i]), v = df_split(o[2 * i + 1]);
      out[i] = make_float4(u.x, u.y, v.x, v.y);
    }
    const float2 f = df_split(o[12]);
    out[6] = make_float4(f.x, f.y, (float)o[13], (float)o[14]);
  } else {
#pragma unroll
    for (int i = 0; i < 15; ++i) rt[15 * (size_t)j + i] = o[i];
  }
}

// F = sum |f_o|^2 at the parameters described by rt and pts (+ dp); writes f_o to rout (working precision).
template <typename real>
__global__ void __launch_bounds__(RED_THREADS) k_cost(DevProblem P, const double* rt, const double* dp,
                                                      double* partial, DevState* st, real* rout) {
  chain_begin();
  double s = 0.0;
  int bad = 0;
  for (int o = blockIdx.x * blockDim.x + threadIdx.x; o < P.q; o += gridDim.x * blockDim.x) {
    const int cam = P.obs_cam[o];
    const int pt = P.obs_pt[o];
    const double* C = rt + 15 * (size_t)cam;
    const double* p = P.pts + 3 * (size_t)pt;
    double X0 = p[0], X1 = p[1], X2 = p[2];
    if (dp) {
      const double* q = dp + 3 * (size_t)pt;
      X0 += q[0];
      X1 += q[1];
      X2 += q[2];
    }
    const double xc = C[0] * X0 + C[1] * X1 + C[2] * X2 + C[9];
    const double yc = C[3] * X0 + C[4] * X1 + C[5] * X2 + C[10];
    const double zc = C[6] * X0 + C[7] * X1 + C[8] * X2 + C[11];
    const double iz = 1.0 / zc;
    const double x = xc * iz, y = yc * iz;
    const double r2 = x * x + y * y;
    const double fd = C[12] * (1.0 + r2 * (C[13] + C[14] * r2));
    const double2 uv = reinterpret_cast<const double2*>(P.obs_uv)[o];
    const double r0 = fd * x - uv.x, r1 = fd * y - uv.y;
    if (!(zc > 1e-9)) bad = 1;
    s += huber_rho(P.huber_a, r0 * r0 + r1 * r1);   // rho(s) = s without a robust loss
    rout[2 * (size_t)o] = (real)r0;
    rout[2 * (size_t)o + 1] = (real)r1;
  }
  __shared__ double buf[1][RED_THREADS];
  if (__any_sync(FULL_MASK, bad) && (threadIdx.x & 31) == 0) st->nonfinite = 1;
  const double v[1] = {s};
  const double a = cta_sums<1>(v, buf);
  if (threadIdx.x == 0) partial[blockIdx.x] = a;
}

// ------------------------------------------------------------------------------------------------------
// Cost of the candidate step in mixed mode, in double-float arithmetic (a value is an unevaluated sum
// hi + lo of two floats, ~48-bit significand; Dekker's and Knuth's error-free transformations, with the
// product error taken by an FMA).  The FP64 pipe of this GPU runs at 1/64 of the FP32 rate; double-float
// keeps the residuals accurate to ~1e-12 px at pixel offsets of a few hundred px on the FP32 pipe.
// Per camera the table of k_cost_cams holds double-float numbers (R, t, f; k1 and k2 as floats, since they
// scale the small distortion term only); per point k_point_update splits the candidate p + dp (k_point_df the
// points of x itself).
__global__ void k_point_df(int n, const double* __restrict__ pts, float2* __restrict__ pdf) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < 3 * n; i += gridDim.x * blockDim.x) pdf[i] = df_split(pts[i]);
}

__global__ void __launch_bounds__(RED_THREADS) k_cost_df(DevProblem P, const float* __restrict__ cdf,
                                                         const float* __restrict__ pdf, double* partial,
                                                         DevState* st, float* rout) {
  chain_begin();
  float2 acc = make_float2(0.f, 0.f);
  double acc_rho = 0.0;
  int bad = 0;
  for (int o = blockIdx.x * blockDim.x + threadIdx.x; o < P.q; o += gridDim.x * blockDim.x) {
    const float4* C4 = reinterpret_cast<const float4*>(cdf + CAM_DF * (size_t)P.obs_cam[o]);
    float cv[CAM_DF];
#pragma unroll
    for (int q4 = 0; q4 < CAM_DF / 4; ++q4) {
      const float4 t4 = __ldg(C4 + q4);
      cv[4 * q4] = t4.x;
      cv[4 * q4 + 1] = t4.y;
      cv[4 * q4 + 2] = t4.z;
      cv[4 * q4 + 3] = t4.w;
    }
    const float2* X2 = reinterpret_cast<const float2*>(pdf) + 3 * (size_t)P.obs_pt[o];
    const float2 X[3] = {X2[0], X2[1], X2[2]};
    float2 Xc[3];
#pragma unroll
    for (int r = 0; r < 3; ++r) {
      const float2 a = df_mul(make_float2(cv[6 * r], cv[6 * r + 1]), X[0]);
      const float2 b = df_mul(make_float2(cv[6 * r + 2], cv[6 * r + 3]), X[1]);
      const float2 c = df_mul(make_float2(cv[6 * r + 4], cv[6 * r + 5]), X[2]);
      Xc[r] = df_add(df_add(a, b), df_add(c, make_float2(cv[18 + 2 * r], cv[19 + 2 * r])));
    }
    if (!(Xc[2].x > 1e-9f)) bad = 1;
    const float2 iz = df_rcp(Xc[2]);
    const float2 x = df_mul(Xc[0], iz), y = df_mul(Xc[1], iz);
    const float r2 = x.x * x.x + y.x * y.x;
    const float2 d = df_fast_two_sum(1.f, r2 * (cv[26] + cv[27] * r2));
    const float2 fd = df_mul(make_float2(cv[24], cv[25]), d);
    const float4 uv = P.obs_uvdf[o];
    const float2 r0 = df_sub(df_mul(fd, x), make_float2(uv.x, uv.y));
    const float2 r1 = df_sub(df_mul(fd, y), make_float2(uv.z, uv.w));
    const float2 sq = df_add(df_mul(r0, r0), df_mul(r1, r1));
    if (P.huber_a > 0.0)   // robust loss: rho of the FP64 value of the double-float square
      acc_rho += huber_rho(P.huber_a, (double)sq.x + (double)sq.y);
    else
      acc = df_add(acc, sq);
    rout[2 * (size_t)o] = r0.x + r0.y;
    rout[2 * (size_t)o + 1] = r1.x + r1.y;
  }
  double s = (double)acc.x + (double)acc.y + acc_rho;
  __shared__ double buf[1][RED_THREADS];
  if (__any_sync(FULL_MASK, bad) && (threadIdx.x & 31) == 0) st->nonfinite = 1;
  const double v[1] = {s};
  const double a = cta_sums<1>(v, buf);
  if (threadIdx.x == 0) partial[blockIdx.x] = a;
}

// ------------------------------------------------------------------------------------------------------
// Stop tests and accept / reject (Algorithm 1), one CTA of one warp per partial sum (fixed order).  32 warps
// took 16 us on the FP64 pipe of the one SM; six warps and paired square roots take 5.3 us.
constexpr int FIN_WARPS = 6;
template <typename real>
__global__ void __launch_bounds__(32 * FIN_WARPS) k_finalize(const double* partial, DevState* st,
                                                             Settings s, int with_step) {
  chain_begin();
  __shared__ double red[FIN_WARPS];
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  constexpr int PER = (RED_BLOCKS + 31) / 32;
  double x[PER];
#pragma unroll
  for (int i = 0; i < PER; ++i) {
    const int e = 32 * i + lane;
    x[i] = e < RED_BLOCKS && (w == 0 || with_step) ? partial[w * RED_BLOCKS + e] : 0.0;
  }
  if (w < FIN_WARPS - 1) {
    double a = x[0], b = x[1];
#pragma unroll
    for (int i = 2; i < PER; i += 2) {
      a += x[i];
      if (i + 1 < PER) b += x[i + 1];
    }
    a += b;
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) a += __shfl_xor_sync(FULL_MASK, a, d);
    if (lane == 0) red[w] = a;
  } else {
    unsigned long long b = 0;
#pragma unroll
    for (int i = 0; i < PER; ++i) {
      const unsigned long long o = (unsigned long long)__double_as_longlong(x[i]);
      b = o > b ? o : b;
    }
    b = warp_max_bits(__longlong_as_double((long long)b));
    if (lane == 0) red[w] = __longlong_as_double((long long)b);
  }
  __syncthreads();
  if (w != 0) return;
  // |dx|^2 = |dp|^2 + |dc|^2 in lane 0, |x|^2 in lane 1: one square root for both
  const double root = sqrt(lane == 0 ? red[1] + red[3] : red[2] + red[4]);
  const double xn = __shfl_sync(FULL_MASK, root, 1);
  if (lane == 0) {
    if (!with_step) {
      st->F = red[0];
      st->info.F_before = red[0];
      return;
    }
    double Fn = red[0];
    const double F = st->F;
    const double lam = st->lambda_used;
    if (st->failed > 0 || st->nonfinite || !isfinite(Fn)) Fn = __longlong_as_double(0x7ff0000000000000ll);
    const double grad = fmax(red[5], __longlong_as_double((long long)st->grad_max_bits));
    const double dxn = root;
    int stop = 0;
    if (s.ftol > 0 && F > 0 && fabs(F - Fn) / F < s.ftol) stop = 1;
    if (s.gtol > 0 && grad < s.gtol) stop = 1;
    if (s.xtol > 0 && dxn < s.xtol * (xn + s.xtol)) stop = 1;
    const int accepted = (Fn < F) ? 1 : 0;
    const double lam_new = accepted ? fmax(lam / 3.0, s.lambda_min) : lam * 3.0;
    st->lambda = lam_new;
    if (accepted) st->F = Fn;
    st->iteration += 1;
    stba_iter_info& I = st->info;
    I.F_before = F;
    I.F_after = Fn;
    I.lambda_used = lam;
    I.lambda = lam_new;
    I.grad_inf = grad;
    I.dx_norm = dxn;
    I.x_norm = xn;
    I.accepted = accepted;
    I.stop = stop;
    I.corrected = st->corrected;
    I.failed_clusters = st->failed;
    I.boosted_pivots = st->boosted;
    I.linear_iterations = 0;
    I.iteration = st->iteration;
  }
}

template <typename real>
__global__ void k_apply(int m, int n, int q, const double* dc, const double* dp, double* cams, double* pts,
                        const real* r_cand, real* r_cur, const DevState* st) {
  chain_begin();
  if (!st->info.accepted) return;
  const int total = 9 * m + 3 * n;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < total; i += gridDim.x * blockDim.x) {
    if (i < 9 * m)
      cams[i] += dc[i];
    else
      pts[i - 9 * m] += dp[i - 9 * m];
  }
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < 2 * q; i += gridDim.x * blockDim.x) r_cur[i] = r_cand[i];
}

// ------------------------------------------------------------------------------------------------------
// launchers
template <typename real>
void launch_point_update(const DevProblem& P, Scratch<real> W, float* pt_df, cudaStream_t stream) {
  launch_after(chained(P), k_point_update<real>, RED_BLOCKS, RED_THREADS, stream, P, W.pt_info, W.t_acc, W.dc, W.vgrad, W.dp,
               reinterpret_cast<float2*>(pt_df), W.partial);
}

template <typename real>
void launch_finalize(const DevProblem& P, const double* partial, DevState* st, const Settings& s, int with_step,
                     cudaStream_t stream) {
  launch_after(chained(P), k_finalize<real>, 1, 32 * FIN_WARPS, stream, partial, st, s, with_step);
}

template <typename real>
void launch_apply(const DevProblem& P, const double* dc, const double* dp, double* cams, double* pts,
                  const real* r_cand, real* r_cur, DevState* st, cudaStream_t stream) {
  int total = std::max(9 * P.m + 3 * P.n, 2 * P.q);
  int blocks = (total + 255) / 256;
  if (blocks > 2048) blocks = 2048;
  launch_after(chained(P), k_apply<real>, blocks, 256, stream, P.m, P.n, P.q, dc, dp, cams, pts, r_cand, r_cur, st);
}

template <typename real>
void launch_point_rhs(const DevProblem& P, Scratch<real> W, cudaStream_t stream) {
  int blocks = (P.q + 255) / 256;
  launch_after(chained(P), k_point_rhs<real>, blocks, 256, stream, P, W.edc, W.t_acc);
}

template <typename real>
void launch_cost_cams(const DevProblem& P, const double* dc, double* rt, float* cam_df, cudaStream_t stream) {
  k_cost_cams<real><<<(P.m + 31) / 32, 32, 0, stream>>>(P.m, P.cams, dc, rt, cam_df);
}

// FP32 working precision: always the double-float kernels (cam_df, pt_df and the double-float observations are
// required; the FP64 observations are not kept in that mode)
template <typename real>
void launch_cost(const DevProblem& P, const double* dp, const double* rt, const float* cam_df, const float* pt_df,
                 double* partial, DevState* st, real* rout, cudaStream_t stream) {
  if constexpr (sizeof(real) == 4)
    k_cost_df<<<RED_BLOCKS, RED_THREADS, 0, stream>>>(P, cam_df, pt_df, partial, st, rout);
  else
    k_cost<real><<<RED_BLOCKS, RED_THREADS, 0, stream>>>(P, rt, dp, partial, st, rout);
}

template <typename real>
void launch_cost_x(const DevProblem& P, double* rt, float* cam_df, float* pt_df, double* partial, DevState* st,
                   real* rout, cudaStream_t stream) {
  launch_cost_cams<real>(P, nullptr, rt, cam_df, stream);
  if constexpr (sizeof(real) == 4)
    k_point_df<<<(int)std::min<int64_t>((3 * (int64_t)P.n + 255) / 256, 2048), 256, 0, stream>>>(
        P.n, P.pts, reinterpret_cast<float2*>(pt_df));
  launch_cost<real>(P, nullptr, rt, cam_df, pt_df, partial, st, rout, stream);
}

// The camera step from the padded cluster vectors x, in the cameras' order, with E dc (edc, if given) and the
// count of failed clusters (st, if given).  sharded: another process's clusters give zeros (their steps arrive
// by the exchange of dc).  One launch for what were three (5.2 + 3.5 + 2.8 us at 1000 cameras, 4.5 us now).
template <typename real>
__global__ void __launch_bounds__(256) k_scatter_step(DevProblem P, const double* x,
                                                      const int* fail_flags, DevState* st,
                                                      const real* ctab, double* __restrict__ dc,
                                                      real* __restrict__ edc) {
  chain_begin();
  const int k = blockIdx.x;
  const int i = blockIdx.y * blockDim.x + threadIdx.x;
  if (st && i == 0 && fail_flags[k] != 0) atomicAdd(&st->failed, 1);
  if (i >= P.cluster_n[k]) return;
  const int cam = P.cluster_cams[P.cluster_cam_off[k] + i / 9], c = i % 9;
  const bool own = !P.sharded || P.cluster_owned[k];
  const double* xc = x + P.v_off[k] + (i - c);
  dc[9 * (size_t)cam + c] = own ? xc[c] : 0.0;
  if (edc) edc[(size_t)VPI * cam + c] = step_entry(jl_ptr(ctab, P.m, cam), xc, c);
}

template <typename real>
void launch_scatter_step(const DevProblem& P, const double* x, const int* fail_flags, int max_np, DevState* st,
                         double* dc, real* edc, cudaStream_t stream) {
  const real* ctab;
  if constexpr (sizeof(real) == 4) ctab = P.ctab_f; else ctab = P.ctab_d;
  launch_after(chained(P), k_scatter_step<real>, dim3(P.l, (max_np + 255) / 256), 256, stream, P, x, fail_flags, st,
               ctab, dc, edc);
}

// The start of an iteration in one launch: the device state, the camera tables (blocks 0 .. cam_blocks - 1, one
// warp each: the FP64 sincos and divisions of a camera run at 1/64 rate, so 32 cameras per SM), in mixed
// precision the FP32 copies of the cameras and points, the zeros of the virtual-point accumulators (9 nv reals,
// nv from the device counter) and of the vectors in Z (the other blocks).  Two kernels, a zeroing kernel and
// four memsets in a row before: linearisation stage 28 -> 17 us at 10 cameras.
template <typename real>
__global__ void __launch_bounds__(256) k_begin(int m, int n, int cam_blocks, const double* __restrict__ cams,
                                               const double* __restrict__ pts, real* __restrict__ ctab,
                                               float* __restrict__ cams_f, float* __restrict__ pts_f, DevState* st,
                                               Settings s, real* __restrict__ vp_acc,
                                               const long long* __restrict__ counts, ZeroList Z) {
  chain_begin();
  if ((int)blockIdx.x < cam_blocks) {
    const int j = 32 * blockIdx.x + threadIdx.x;
    if (threadIdx.x < 32 && j < m) write_camtab<real>(cams + 9 * (size_t)j, m, j, ctab);
    if (blockIdx.x == 0 && threadIdx.x == 32) reset_state(st, s);
    return;
  }
  const int64_t first = ((int64_t)blockIdx.x - cam_blocks) * blockDim.x + threadIdx.x;
  const int64_t step = ((int64_t)gridDim.x - cam_blocks) * blockDim.x;
  const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
  const int64_t nz = (9 * counts[0] * (int64_t)sizeof(real) + 15) / 16;   // the buffer is padded to 16 bytes
  for (int64_t i = first; i < nz; i += step) reinterpret_cast<float4*>(vp_acc)[i] = zero;
#pragma unroll
  for (int z = 0; z < ZeroList::N; ++z)
    for (int64_t i = first; i < Z.words[z]; i += step) Z.p[z][i] = 0;
  if (cams_f) {
    for (int64_t i = first; i < 9 * (int64_t)m; i += step) cams_f[i] = (float)cams[i];
    for (int64_t i = first; i < 3 * (int64_t)n; i += step) pts_f[i] = (float)pts[i];
  }
}

template <typename real>
void launch_begin(const DevProblem& P, Scratch<real> W, real* ctab, float* cams_f, float* pts_f, DevState* st,
                  const Settings& s, const long long* counts, const ZeroList& Z, cudaStream_t stream) {
  const int cam_blocks = (P.m + 31) / 32;
  int64_t work = 9 * (int64_t)P.m + 3 * (int64_t)P.n;
  for (int z = 0; z < ZeroList::N; ++z) work = std::max<int64_t>(work, Z.words[z]);
  const int rest = (int)std::min<int64_t>((work + 255) / 256, 8 * (int64_t)num_sms());
  k_begin<real><<<cam_blocks + rest, 256, 0, stream>>>(P.m, P.n, cam_blocks, P.cams, P.pts, ctab, cams_f, pts_f, st, s,
                                                       W.vp_acc, counts, Z);
}

void configure_kernels(int max_np) {
  configure_solve_kernels(max_np);
  cudaFuncSetAttribute(k_pair_build<float, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                       (int)PairRows<float>::bytes);
  cudaFuncSetAttribute(k_pair_build<float, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                       (int)PairRows<float>::bytes);
  cudaFuncSetAttribute(k_pair_build<double, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                       (int)PairRows<double>::bytes);
  cudaFuncSetAttribute(k_pair_build<double, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                       (int)PairRows<double>::bytes);
}

#define INSTANTIATE(real)                                                                                  \
  template void launch_begin<real>(const DevProblem&, Scratch<real>, real*, float*, float*, DevState*,    \
                                   const Settings&, const long long*, const ZeroList&, cudaStream_t);     \
  template void launch_vp_reduce<real>(const DevProblem&, Scratch<real>, cudaStream_t);                   \
  template void launch_vp_finalize<real>(const DevProblem&, Scratch<real>, DevState*, const long long*,   \
                                         cudaStream_t, const double*);                                     \
  template void launch_pt_sums<real>(const DevProblem&, Scratch<real>, double*, cudaStream_t);              \
  template void launch_rcs_build<real>(const DevProblem&, Scratch<real>, CamSlots, PairChunks, real*,     \
                                       DevState*, cudaStream_t, cudaStream_t, cudaEvent_t, cudaEvent_t);  \
  template void launch_scatter_step<real>(const DevProblem&, const double*, const int*, int, DevState*,   \
                                          double*, real*, cudaStream_t);                                  \
  template void launch_point_update<real>(const DevProblem&, Scratch<real>, float*, cudaStream_t);        \
  template void launch_finalize<real>(const DevProblem&, const double*, DevState*, const Settings&, int,  \
                                      cudaStream_t);                                                      \
  template void launch_step_rows<real>(const DevProblem&, const double*, real*, cudaStream_t);            \
  template void launch_point_rhs<real>(const DevProblem&, Scratch<real>, cudaStream_t);                  \
  template void launch_cost_cams<real>(const DevProblem&, const double*, double*, float*, cudaStream_t);  \
  template void launch_cost<real>(const DevProblem&, const double*, const double*, const float*,          \
                                  const float*, double*, DevState*, real*, cudaStream_t);                 \
  template void launch_cost_x<real>(const DevProblem&, double*, float*, float*, double*, DevState*, real*, \
                                    cudaStream_t);                                                        \
  template void launch_apply<real>(const DevProblem&, const double*, const double*, double*, double*,     \
                                   const real*, real*, DevState*, cudaStream_t);

INSTANTIATE(float)
INSTANTIATE(double)

}  // namespace stba
