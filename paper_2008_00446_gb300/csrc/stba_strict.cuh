// FP32 numbers whose rounding is fixed by the source: a product is held unrounded (SFProd) and fused with
// the addition or subtraction it meets (one fused multiply-add, __fmaf_rn), every other operation is rounded
// on its own (__fadd_rn, __fmul_rn, ...), and the compiler contracts or re-associates nothing.  The
// arithmetic of an expression is then the same in every kernel that evaluates it.  The FP32 kernels that form
// V_v, the diagonal and the off-diagonal blocks of S'_k (Eq. 10, 13) all evaluate the reprojection Jacobian
// of an observation (Sec. 3; stba_camtab.cuh) on this type, so that they see bitwise the same rows, whether the
// pair pass reads the camera pass's copy or recomputes it.
#pragma once
#include <cuda_runtime.h>

#include "stba_camera.cuh"

namespace stba {

struct SFProd;

struct SF {
  float v;
  SF() = default;
  __host__ __device__ constexpr SF(float x) : v(x) {}
  __device__ __forceinline__ SF(const SFProd& p);   // the product, rounded

  friend __device__ __forceinline__ SF operator+(SF a, SF b) { return SF(__fadd_rn(a.v, b.v)); }
  friend __device__ __forceinline__ SF operator-(SF a, SF b) { return SF(__fsub_rn(a.v, b.v)); }
  friend __device__ __forceinline__ SF operator-(SF a) { return SF(-a.v); }
  friend __device__ __forceinline__ SFProd operator*(SF a, SF b);
};

// a * b, not yet rounded
struct SFProd {
  float a, b;
  __device__ __forceinline__ float rounded() const { return __fmul_rn(a, b); }

  friend __device__ __forceinline__ SF operator+(SFProd p, SF c) { return SF(__fmaf_rn(p.a, p.b, c.v)); }
  friend __device__ __forceinline__ SF operator+(SF c, SFProd p) { return SF(__fmaf_rn(p.a, p.b, c.v)); }
  friend __device__ __forceinline__ SF operator+(SFProd p, SFProd q) { return SF(__fmaf_rn(p.a, p.b, q.rounded())); }
  friend __device__ __forceinline__ SF operator-(SFProd p, SF c) { return SF(__fmaf_rn(p.a, p.b, -c.v)); }
  friend __device__ __forceinline__ SF operator-(SF c, SFProd p) { return SF(__fmaf_rn(-p.a, p.b, c.v)); }
  friend __device__ __forceinline__ SF operator-(SFProd p, SFProd q) { return SF(__fmaf_rn(p.a, p.b, -q.rounded())); }
  friend __device__ __forceinline__ SFProd operator-(SFProd p) { return SFProd{-p.a, p.b}; }
  friend __device__ __forceinline__ SFProd operator*(SFProd p, SF c) { return SFProd{p.rounded(), c.v}; }
  friend __device__ __forceinline__ SFProd operator*(SF c, SFProd p) { return SFProd{c.v, p.rounded()}; }
  friend __device__ __forceinline__ SFProd operator*(SFProd p, SFProd q) { return SFProd{p.rounded(), q.rounded()}; }
};

__device__ __forceinline__ SF::SF(const SFProd& p) : v(p.rounded()) {}
__device__ __forceinline__ SFProd operator*(SF a, SF b) { return SFProd{a.v, b.v}; }

// sqrt(rho'(|f|^2)) of the Huber loss (1 without a robust loss), every operation rounded on its own.
__device__ __forceinline__ float huber_sqrt_weight_strict(double a, float r0, float r1) {
  if (!(a > 0.0)) return 1.f;
  const float s = __fadd_rn(__fmul_rn(r0, r0), __fmul_rn(r1, r1)), ar = (float)a;
  return s <= __fmul_rn(ar, ar) ? 1.f : __fsqrt_rn(__fdiv_rn(ar, __fsqrt_rn(s)));
}

}  // namespace stba
