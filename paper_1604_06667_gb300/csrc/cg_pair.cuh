// cg_pair.cuh -- pieces shared by the FP32 gridders and the adjoint: the
// kernel's exponential, compensated sums, and the weights of pairs on packed
// f32x2 lanes.
#pragma once
#include <cuda_runtime.h>

#include "cg_common.cuh"
#include "cg_internal.h"

namespace cg {
namespace {

__device__ __forceinline__ float ex2_approx(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

__host__ __device__ __forceinline__ float2 f2(float x) { return make_float2(x, x); }

// Factor of a target's map row in the adjoint: 1 / W_p (0 where W_p <= 0 or not
// finite) from a user-order weight map or the slot-order accumulator;
// interpolation: 1.
__device__ __forceinline__ float target_factor(uint32_t slot, uint32_t user,
                                               const float* __restrict__ wmap,
                                               const float2* __restrict__ acc_w, int interp) {
  if (user == 0xffffffffu) return 0.f;
  if (interp) return 1.f;
  float W;
  if (wmap) {
    W = wmap[user];
  } else {
    const float2 a = acc_w[slot];
    W = a.x + a.y;
  }
  return (W > 0.f && isfinite(W)) ? 1.f / W : 0.f;
}

// (s, c) + (v, vc): two-sum of the leading parts, the corrections added up.
__device__ __forceinline__ void comp_add(float& s, float& c, float v, float vc) {
  const float t = s + v;
  const float b = t - s;
  c += (s - (t - b)) + (v - b) + vc;
  s = t;
}

// Kahan sums of two lanes: s += w with the correction nc (the negative of what
// is still to subtract); the differences as fma with -1, since packed operands
// take no sign.
__device__ __forceinline__ void kahan2(float2& s, float2& nc, float2 w) {
  const float2 m1 = make_float2(-1.f, -1.f);
  const float2 y = __fadd2_rn(w, nc);
  const float2 t = __fadd2_rn(s, y);
  const float2 e = __ffma2_rn(s, m1, t);
  nc = __ffma2_rn(e, m1, y);
  s = t;
}

// Distance of two squared chords from the centre of the guard band, the smaller
// with what came before.
__device__ __forceinline__ float band_near(const WeightConst& k, float2 c2, float before) {
  const float2 x = __fadd2_rn(c2, k.nmid);
  return fminf(fminf(fabsf(x.x), fabsf(x.y)), before);
}

// Forms of the weight evaluation: the Gaussians with the series for d^2 (c^2
// small, see KernelDev::big_support), the circular one's width derivative, and
// everything else (large supports, the tapered sinc) chosen at run time.
enum { kWGauss1 = 0, kWGauss2 = 1, kWAny = 2, kWGauss1Ds = 3 };
inline int weight_form(const KernelDev& kd) {
  if (kd.big_support || kd.type == CG_TSINC) return kWAny;
  if (kd.dscale != 0.f) return kd.type == CG_GAUSS1D ? kWGauss1Ds : kWAny;
  return kd.type == CG_GAUSS1D ? kWGauss1 : kWGauss2;
}

__host__ __device__ __forceinline__ WeightConst weight_const(const KernelDev& kd) {
  WeightConst c;
  c.q0 = f2(kd.k1);
  c.q1 = f2(kd.k1 * (1.f / 12.f));
  c.q2 = f2(kd.k1 * (1.f / 90.f));
  c.k1 = f2(kd.k1);
  c.k2 = f2(kd.k2);
  c.ds = f2(kd.dscale / kd.k1);
  c.c2_out = kd.c2_out;
  // (a little wide: the sum and difference round; who falls in here is decided
  // against c2_in and c2_out themselves)
  const float mid = 0.5f * (kd.c2_in + kd.c2_out);
  c.nmid = f2(-mid);
  c.hw = 0.5f * (kd.c2_out - kd.c2_in) * 1.02f;
  return c;
}

// Kernel value (without sample weight, cut not applied) of one pair: squared
// chord c2, difference vector d, major / minor axis directions f1, f2.
__device__ __forceinline__ float weight_any(const KernelDev& kd, float c2, float3 d, float3 f1,
                                            float3 f2v) {
  float d2;
  if (!kd.big_support) {
    d2 = c2 * fmaf(c2, fmaf(c2, 1.f / 90.f, 1.f / 12.f), 1.f);
  } else {
    const float ang = 2.f * asinf(fminf(1.f, 0.5f * sqrtf(c2)));
    d2 = ang * ang;
  }
  float ex;
  if (kd.type == CG_GAUSS1D || kd.type == CG_TSINC) {
    ex = kd.k1 * d2;
  } else {
    const float ap = fmaf(d.x, f1.x, fmaf(d.y, f1.y, d.z * f1.z));
    const float bp = fmaf(d.x, f2v.x, fmaf(d.y, f2v.y, d.z * f2v.z));
    const float s2 = fmaf(ap, ap, bp * bp);  // sin^2 d
    const float ratio = (s2 > 0.f) ? __fdividef(d2, s2) : 1.f;
    ex = fmaf(kd.k1 * ap, ap, kd.k2 * bp * bp) * ratio;
  }
  float w = ex2_approx(ex);
  if (kd.type == CG_TSINC) w *= sinc_pi(sqrtf(d2) * kd.inv_a);
  if (kd.dscale != 0.f) w *= d2 * kd.dscale;   // dw/dsigma pass
  return w;
}

// Axis directions of two targets, packed.
struct Axes2 {
  float2 ax, ay, az, bx, by, bz;
};

// Kernel values of two pairs (packed lanes): squared chords c2, differences
// (dx, dy, dz).  The elliptical form uses (d / sin d)^2 = 1 + c^2 / 3 + 17
// c^4 / 180 (the next term is below 4e-8 for c <= 0.1).
template <int FORM>
__device__ __forceinline__ float2 weight2(const WeightConst& k, const KernelDev& kd, float2 c2,
                                          float2 dx, float2 dy, float2 dz, const Axes2& A) {
  if constexpr (FORM == kWGauss1) {
    const float2 e = __fmul2_rn(c2, __ffma2_rn(c2, __ffma2_rn(c2, k.q2, k.q1), k.q0));
    return make_float2(ex2_approx(e.x), ex2_approx(e.y));
  } else if constexpr (FORM == kWGauss1Ds) {
    const float2 e = __fmul2_rn(c2, __ffma2_rn(c2, __ffma2_rn(c2, k.q2, k.q1), k.q0));
    return __fmul2_rn(__fmul2_rn(e, k.ds), make_float2(ex2_approx(e.x), ex2_approx(e.y)));
  } else if constexpr (FORM == kWGauss2) {
    const float2 ap = __ffma2_rn(dx, A.ax, __ffma2_rn(dy, A.ay, __fmul2_rn(dz, A.az)));
    const float2 bp = __ffma2_rn(dx, A.bx, __ffma2_rn(dy, A.by, __fmul2_rn(dz, A.bz)));
    const float2 ratio = __ffma2_rn(c2, __ffma2_rn(c2, f2(17.f / 180.f), f2(1.f / 3.f)), f2(1.f));
    const float2 t = __ffma2_rn(__fmul2_rn(k.k1, ap), ap, __fmul2_rn(__fmul2_rn(k.k2, bp), bp));
    const float2 e = __fmul2_rn(t, ratio);
    return make_float2(ex2_approx(e.x), ex2_approx(e.y));
  } else {
    return make_float2(
        weight_any(kd, c2.x, make_float3(dx.x, dy.x, dz.x), make_float3(A.ax.x, A.ay.x, A.az.x),
                   make_float3(A.bx.x, A.by.x, A.bz.x)),
        weight_any(kd, c2.y, make_float3(dx.y, dy.y, dz.y), make_float3(A.ax.y, A.ay.y, A.az.y),
                   make_float3(A.bx.y, A.by.y, A.bz.y)));
  }
}

}  // namespace
}  // namespace cg
