// tt_f2.cuh -- compensated fp32 pairs (an unevaluated sum hi + lo, about
// 2^-44 relative), 2^y with an exact exponent split, and the grid-dependency
// wait, shared by the decision kernels (decide.cu, filter.cu).
#pragma once

#include "tt_device.cuh"

namespace tt {

struct F2 {  // unevaluated sum hi + lo
  float hi, lo;
};

__device__ __forceinline__ F2 two_sum(float a, float b) {
  const float s = __fadd_rn(a, b);
  const float bb = __fsub_rn(s, a);
  return {s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb))};
}

__device__ __forceinline__ F2 f2_add(F2 a, F2 b) {
  const F2 s = two_sum(a.hi, b.hi);
  const float lo = __fadd_rn(s.lo, __fadd_rn(a.lo, b.lo));
  const float hi = __fadd_rn(s.hi, lo);
  return {hi, __fsub_rn(lo, __fsub_rn(hi, s.hi))};
}

// a * b as a normalised pair.
__device__ __forceinline__ F2 f2_mul_f(F2 a, float b) {
  const float p = __fmul_rn(a.hi, b);
  const float e = fmaf(a.hi, b, -p);
  const float lo = fmaf(a.lo, b, e);
  const float hi = __fadd_rn(p, lo);
  return {hi, __fsub_rn(lo, __fsub_rn(hi, p))};
}

__device__ __forceinline__ bool f2_lt(F2 a, F2 b) {
  return a.hi < b.hi || (a.hi == b.hi && a.lo < b.lo);
}

__device__ __forceinline__ F2 shfl_up_f2(F2 v, int o, int width = 32) {
  return {__shfl_up_sync(0xffffffffu, v.hi, o, width), __shfl_up_sync(0xffffffffu, v.lo, o, width)};
}

// 2^(z * scale - M) with the exponent split exactly (TwoProd, TwoSum, rint);
// only 2^f, |f| <= 1/2, comes from the SFU.
__device__ __forceinline__ float exp2_scaled(float z, float scale, float M) {
  const float xh = __fmul_rn(z, scale);
  const float xl = fmaf(z, scale, -xh);
  const F2 d = two_sum(xh, -M);
  const float n = rintf(d.hi);
  const float f = __fadd_rn(__fsub_rn(d.hi, n), __fadd_rn(d.lo, xl));
  if (!(n > -126.f)) return 0.f;
  return ex2_approx(f) * __int_as_float((int(n) + 127) << 23);
}

// The normaliser of a nucleus row from its kept mass `tot` (40-bit fixed point,
// relative to 2^M): 2^40 / tot and the natural log of tot 2^(M - 40), from fp32
// pairs (about an ulp; fp64 is slow here). Every kernel that settles nucleus
// rows forms them this way, so that a row's result does not depend on which did.
constexpr float kFixScale = 1099511627776.f;  // 2^40
struct KeptNorm {
  float inv_tot, inv_s, lse;  // 1 / tot, 2^40 / tot
};
__device__ __forceinline__ KeptNorm kept_norm(unsigned long long tot, float M) {
  const float sh = __ull2float_rn(tot);
  const float sl = __ll2float_rn((long long)(tot - __float2ull_rn(sh)));
  const float r = __frcp_rn(sh);
  const float inv = fmaf(r, fmaf(-sl, r, fmaf(-sh, r, 1.f)), r);
  const F2 l2 = two_sum(M, log2f(sh * (1.f / kFixScale)));
  const float ln2 = 0.693147180559945f, ln2l = 1.904654299957768e-9f;
  const float ph = __fmul_rn(l2.hi, ln2);
  const float pl = fmaf(l2.hi, ln2, -ph) + fmaf(l2.hi, ln2l, l2.lo * ln2);
  return {inv, inv * kFixScale, ph + pl};
}

__device__ __forceinline__ void grid_dependency_wait() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
}

}  // namespace tt
