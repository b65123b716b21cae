// Per-camera tables of the reprojection Jacobian (Sec. 3).  The rotation of a camera and its derivative do not
// depend on the observation, so they are formed once per camera and linearisation -- R(w) and the left Jacobian
// Jl(w) of the rotation group, in FP64, rounded to the working precision -- and every per-observation kernel
// works from them without trigonometry or divisions (one reciprocal of the depth):
//   Y = R X, Xc = Y + t, P = d pi / d Xc (2x3);  d pi / d t = P, d pi / d X = P R,
//   d(R X) / d w = -[Y]x Jl(w)   =>   row s of d pi / d w = (Y x P_s)^T Jl(w).
// The rows before the factor Jl, (Y x P_s | P_s | d pi_s / d(f, k1, k2)), are the "tilde" rows: J_c = Jt E with
// E = diag(Jl, I, I) a constant of the camera.
// About 100 multiply-adds per observation; evaluating Rodrigues' formula and its derivative per observation
// took about 350 instructions (two sincos, divisions by |w|^2).  FP32: the operations on SF numbers
// (stba_strict.cuh), so that every kernel sees bitwise the same rows.
#pragma once
#include "stba_device.cuh"
#include "stba_internal.cuh"
#include "stba_strict.cuh"

namespace stba {

// Three tables, one after the other, 16-byte aligned records:
//   R (9), t (3), f, k1, k2, -          [m][16]  kernels whose warps work on one camera (or two)
//   q (4), t (3), f, k1, k2, -, -       [m][12]  kernels that gather a camera per lane: the rotation as a unit
//                                                quaternion in 48 bytes (three 16-byte loads, and 1000 cameras
//                                                stay in L1); R(q) is the same arithmetic in both
//   Jl (9), -, -, -                     [m][12]
constexpr int CTAB_R = 16, CTAB_Q = 12, CTAB_L = 12, CTAB = CTAB_R + CTAB_Q + CTAB_L;

template <typename real> __device__ __forceinline__ const real* ctab_ptr(const DevProblem& P);
template <> __device__ __forceinline__ const float* ctab_ptr<float>(const DevProblem& P) { return P.ctab_f; }
template <> __device__ __forceinline__ const double* ctab_ptr<double>(const DevProblem& P) { return P.ctab_d; }

// number type of the per-observation arithmetic
template <typename real> struct RowNum;
template <> struct RowNum<float> { using T = SF; };
template <> struct RowNum<double> { using T = double; };

__device__ __forceinline__ SF rcp_num(SF a) { return SF(__frcp_rn(a.v)); }
__device__ __forceinline__ double rcp_num(double a) { return __drcp_rn(a); }

// N reals (a multiple of 16 bytes) from a 16-byte aligned address through the read-only path: for kernels that are
// not chained (chain_begin)
template <int N, typename real>
__device__ __forceinline__ void load_vec16(const real* p, real (&v)[N]) {
  if constexpr (sizeof(real) == 4) {
#pragma unroll
    for (int k = 0; k < N / 4; ++k) {
      const float4 t = __ldg(reinterpret_cast<const float4*>(p) + k);
      v[4 * k] = t.x;
      v[4 * k + 1] = t.y;
      v[4 * k + 2] = t.z;
      v[4 * k + 3] = t.w;
    }
  } else {
#pragma unroll
    for (int k = 0; k < N / 2; ++k) {
      const double2 t = __ldg(reinterpret_cast<const double2*>(p) + k);
      v[2 * k] = t.x;
      v[2 * k + 1] = t.y;
    }
  }
}

// the same with ordinary loads: for chained kernels too
template <int N, typename real>
__device__ __forceinline__ void gather_vec16(const real* p, real (&v)[N]) {
  if constexpr (sizeof(real) == 4) {
#pragma unroll
    for (int k = 0; k < N / 4; ++k) {
      const float4 t = reinterpret_cast<const float4*>(p)[k];
      v[4 * k] = t.x;
      v[4 * k + 1] = t.y;
      v[4 * k + 2] = t.z;
      v[4 * k + 3] = t.w;
    }
  } else {
#pragma unroll
    for (int k = 0; k < N / 2; ++k) {
      const double2 t = reinterpret_cast<const double2*>(p)[k];
      v[2 * k] = t.x;
      v[2 * k + 1] = t.y;
    }
  }
}

// R(q) of a unit quaternion (row-major)
template <typename T>
__device__ __forceinline__ void quat_rotation(const T (&q)[4], T (&R)[9]) {
  const T x2 = q[1] + q[1], y2 = q[2] + q[2], z2 = q[3] + q[3];
  const T xx = q[1] * x2, wx = q[0] * x2, wy = q[0] * y2, wz = q[0] * z2;
  R[0] = T(1) - T(q[2] * y2 + q[3] * z2);
  R[4] = T(1) - T(q[3] * z2 + xx);
  R[8] = T(1) - T(q[2] * y2 + xx);
  R[1] = q[1] * y2 - wz;
  R[3] = q[1] * y2 + wz;
  R[2] = q[1] * z2 + wy;
  R[6] = q[1] * z2 - wy;
  R[5] = q[2] * z2 - wx;
  R[7] = q[2] * z2 + wx;
}

// R, t, f, k1, k2 of camera j: v[0..8], v[9..11], v[12..14]
template <typename real> struct CamRow {
  real v[16];
};
template <typename real>
__device__ __forceinline__ CamRow<real> load_camrow(const DevProblem& P, int j) {
  CamRow<real> C;
  load_vec16<16>(ctab_ptr<real>(P) + (size_t)CTAB_R * j, C.v);
  return C;
}
// the same from the quaternion record (for lanes of different cameras)
template <typename real>
__device__ __forceinline__ CamRow<real> gather_camrow(const DevProblem& P, int j) {
  using T = typename RowNum<real>::T;
  real v[12];
  gather_vec16<12>(ctab_ptr<real>(P) + (size_t)CTAB_R * P.m + (size_t)CTAB_Q * j, v);
  const T q[4] = {T(v[0]), T(v[1]), T(v[2]), T(v[3])};
  T Rm[9];
  quat_rotation(q, Rm);
  CamRow<real> C;
#pragma unroll
  for (int i = 0; i < 9; ++i)
    if constexpr (sizeof(real) == 4) C.v[i] = Rm[i].v; else C.v[i] = Rm[i];
#pragma unroll
  for (int i = 0; i < 6; ++i) C.v[9 + i] = v[4 + i];
  C.v[15] = real(0);
  return C;
}
// Jl of camera j, row-major
template <typename real>
__device__ __forceinline__ const real* jl_ptr(const real* ctab, int m, int j) {
  return ctab + (size_t)(CTAB_R + CTAB_Q) * m + (size_t)CTAB_L * j;
}
template <typename real>
__device__ __forceinline__ void load_jl(const DevProblem& P, int j, real (&Jl)[9]) {
  real t[12];
  load_vec16<12>(jl_ptr(ctab_ptr<real>(P), P.m, j), t);
#pragma unroll
  for (int i = 0; i < 9; ++i) Jl[i] = t[i];
}
// entry c of E dc for one camera's step (9 entries): J_c dc = Jt (E dc)
template <typename real>
__device__ __forceinline__ real step_entry(const real* Jl, const double* dc, int c) {
  if (c >= 3) return (real)dc[c];
  return (real)((double)Jl[3 * c] * dc[0] + (double)Jl[3 * c + 1] * dc[1] + (double)Jl[3 * c + 2] * dc[2]);
}

// The point rows Jp (2x3) and, with CAM, the tilde rows Jt (2x9) of one observation.
template <typename real, bool CAM>
__device__ __forceinline__ void proj_rows(const CamRow<real>& Cr, const real (&Xr)[3], real (&Jt)[2][9], real (&Jp)[2][3]) {
  using T = typename RowNum<real>::T;
  T R[9];
#pragma unroll
  for (int i = 0; i < 9; ++i) R[i] = T(Cr.v[i]);
  const T f(Cr.v[12]), k1(Cr.v[13]), k2(Cr.v[14]);
  T Y[3], Xc[3];
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    Y[i] = R[3 * i] * T(Xr[0]) + R[3 * i + 1] * T(Xr[1]) + R[3 * i + 2] * T(Xr[2]);
    Xc[i] = Y[i] + T(Cr.v[9 + i]);
  }
  const T iz = rcp_num(Xc[2]);
  const T x = Xc[0] * iz, y = Xc[1] * iz;
  const T r2 = x * x + y * y;
  const T kr = k1 + k2 * r2;
  const T d = T(real(1)) + r2 * kr;
  const T fd = f * d;
  const T e = kr + k2 * r2;              // k1 + 2 k2 r2
  const T fe = f * e;
  const T fe2 = fe + fe;
  const T fx = fe2 * x, fy = fe2 * y;
  const T dux = fd + fx * x, duy = fx * y, dvy = fd + fy * y;
  T Pm[2][3];
  Pm[0][0] = dux * iz;
  Pm[0][1] = duy * iz;
  Pm[1][0] = Pm[0][1];
  Pm[1][1] = dvy * iz;
  Pm[0][2] = -(Pm[0][0] * x + Pm[0][1] * y);
  Pm[1][2] = -(Pm[1][0] * x + Pm[1][1] * y);
#pragma unroll
  for (int s = 0; s < 2; ++s)
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      const T v = Pm[s][0] * R[j] + Pm[s][1] * R[3 + j] + Pm[s][2] * R[6 + j];
      if constexpr (sizeof(real) == 4) Jp[s][j] = v.v; else Jp[s][j] = v;
    }
  if constexpr (CAM) {
    const T fr2 = f * r2;
    const T fr4 = fr2 * r2;
    T J[2][9];
#pragma unroll
    for (int s = 0; s < 2; ++s) {
      J[s][0] = Y[1] * Pm[s][2] - Y[2] * Pm[s][1];
      J[s][1] = Y[2] * Pm[s][0] - Y[0] * Pm[s][2];
      J[s][2] = Y[0] * Pm[s][1] - Y[1] * Pm[s][0];
      J[s][3] = Pm[s][0];
      J[s][4] = Pm[s][1];
      J[s][5] = Pm[s][2];
      const T xs = s ? y : x;
      J[s][6] = d * xs;
      J[s][7] = fr2 * xs;
      J[s][8] = fr4 * xs;
#pragma unroll
      for (int c = 0; c < 9; ++c)
        if constexpr (sizeof(real) == 4) Jt[s][c] = J[s][c].v; else Jt[s][c] = J[s][c];
    }
  }
}

// the first three columns of the tilde rows times Jl: the camera rows J_c
template <typename real>
__device__ __forceinline__ void apply_jl(const real (&Jl)[9], real (&J)[2][9]) {
  using T = typename RowNum<real>::T;
#pragma unroll
  for (int s = 0; s < 2; ++s) {
    const T a(J[s][0]), b(J[s][1]), c(J[s][2]);
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      const T v = a * T(Jl[j]) + b * T(Jl[3 + j]) + c * T(Jl[6 + j]);
      if constexpr (sizeof(real) == 4) J[s][j] = v.v; else J[s][j] = v;
    }
  }
}

// sqrt(rho') of the Huber loss at the residual r
template <typename real>
__device__ __forceinline__ real row_weight(const DevProblem& P, real r0, real r1) {
  if constexpr (sizeof(real) == 4)
    return huber_sqrt_weight_strict(P.huber_a, r0, r1);
  else
    return huber_sqrt_weight<real>(P.huber_a, r0, r1);
}

// The table records of camera j: q(w) and Jl(w) = I + b [w]x + c [w]x^2 in FP64, b = (1 - cos th) / th^2,
// c = (th - sin th) / th^3; series in s = th^2 near zero.
template <typename real>
__device__ __forceinline__ void write_camtab(const double* __restrict__ cam, int m, int j, real* __restrict__ ctab) {
  using T = typename RowNum<real>::T;
  double w[9];
#pragma unroll
  for (int i = 0; i < 9; ++i) w[i] = cam[i];
  const double s = w[0] * w[0] + w[1] * w[1] + w[2] * w[2];
  double b, c, qw, qs;   // q = (qw, qs w)
  if (s < RodSeries<double>::cut) {
    b = 0.5 - s * (1.0 / 24 - s * (1.0 / 720 - s * (1.0 / 40320)));
    c = 1.0 / 6 - s * (1.0 / 120 - s * (1.0 / 5040 - s * (1.0 / 362880)));
    qw = 1.0 - s * (1.0 / 8 - s * (1.0 / 384 - s * (1.0 / 46080)));
    qs = 0.5 - s * (1.0 / 48 - s * (1.0 / 3840 - s * (1.0 / 645120)));
  } else {
    // sin and cos of the half angle: sin th = 2 sh ch, 1 - cos th = 2 sh^2
    const double th = sqrt(s), is = 1.0 / s;
    double sh;
    sincos(0.5 * th, &sh, &qw);
    qs = sh * th * is;
    b = 2.0 * sh * sh * is;
    c = (1.0 - 2.0 * qw * qs) * is;
  }
  const real q[4] = {(real)qw, (real)(qs * w[0]), (real)(qs * w[1]), (real)(qs * w[2])};
  const T qt[4] = {T(q[0]), T(q[1]), T(q[2]), T(q[3])};
  T Rm[9];
  quat_rotation(qt, Rm);
  real* r = ctab + (size_t)CTAB_R * j;
  real* rq = ctab + (size_t)CTAB_R * m + (size_t)CTAB_Q * j;
  real* rl = ctab + (size_t)(CTAB_R + CTAB_Q) * m + (size_t)CTAB_L * j;
#pragma unroll
  for (int i = 0; i < 9; ++i)
    if constexpr (sizeof(real) == 4) r[i] = Rm[i].v; else r[i] = Rm[i];
#pragma unroll
  for (int i = 0; i < 4; ++i) rq[i] = q[i];
#pragma unroll
  for (int i = 0; i < 6; ++i) {
    r[9 + i] = (real)w[3 + i];
    rq[4 + i] = (real)w[3 + i];
  }
  r[15] = rq[10] = rq[11] = real(0);
  const double xx = w[0] * w[0], yy = w[1] * w[1], zz = w[2] * w[2], xy = w[0] * w[1], xz = w[0] * w[2],
               yz = w[1] * w[2];
  const double v[9] = {1.0 - c * (yy + zz), c * xy - b * w[2], c * xz + b * w[1],
                       c * xy + b * w[2], 1.0 - c * (xx + zz), c * yz - b * w[0],
                       c * xz - b * w[1], c * yz + b * w[0], 1.0 - c * (xx + yy)};
#pragma unroll
  for (int i = 0; i < 9; ++i) rl[i] = (real)v[i];
  rl[9] = rl[10] = rl[11] = real(0);
}

}  // namespace stba
