// tt_f2.cuh -- compensated fp32 pairs (an unevaluated sum hi + lo, about
// 2^-44 relative), 2^y with an exact exponent split, the normaliser of a nucleus
// row's kept set, and the grid-dependency wait: shared by the kernels of all
// stages.
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

// Adds m to a 64-bit sum in shared memory by 32-bit adds, the carry from the lower
// word's old value (the sum is whole once all adds are done: read it past a
// barrier). A 64-bit atomicAdd is a loop around compare-and-swap there, and lanes
// that meet at one sum, as the candidates of a region do at one chunk, go round
// it in turn: 64 requests of 151,936 fp32 columns whose rows need the histogram
// levels (Gaussian logits, sigma 1, top-p 0.9) take 1562 us a step, 2792 with it.
__device__ __forceinline__ void shared_add_u64(unsigned long long* sum, unsigned long long m) {
  unsigned int* w = reinterpret_cast<unsigned int*>(sum);
  const unsigned int lo = static_cast<unsigned int>(m), old = atomicAdd(w, lo);
  const unsigned int hi = static_cast<unsigned int>(m >> 32) + (old + lo < old ? 1u : 0u);
  if (hi) atomicAdd(w + 1, hi);
}

// The kept set of a nucleus row from its kept mass `tot` (40-bit fixed point,
// relative to 2^M). Every kernel that settles nucleus rows forms these the same
// way, so that a row's result does not depend on which did.
constexpr float kFixScale = 1099511627776.f;  // 2^40
// A chunk's share c / tot of it, from fp32 pairs (about half an ulp; a division
// in fp64, which is slow here, for each chunk of every row held the cuts up).
struct KeptNorm {
  float hi, lo, inv;  // tot = hi + lo; 1 / tot
};
__device__ __forceinline__ KeptNorm kept_norm(unsigned long long tot) {
  const float hi = __ull2float_rn(tot);
  const float lo = __ll2float_rn((long long)(tot - __float2ull_rn(hi)));
  const float r = __frcp_rn(hi);
  return {hi, lo, fmaf(r, fmaf(-lo, r, fmaf(-hi, r, 1.f)), r)};
}
__device__ __forceinline__ float kept_share(unsigned long long c, const KeptNorm& k) {
  const float hi = __ull2float_rn(c);
  const float lo = __ll2float_rn((long long)(c - __float2ull_rn(hi)));
  const float q = __fmul_rn(hi, k.inv);
  return fmaf(__fadd_rn(fmaf(-q, k.hi, hi), fmaf(-q, k.lo, lo)), k.inv, q);
}
// The natural log of the normaliser sum, and 2^40 / tot. log(m 2^e) = e log 2 +
// 2 atanh((m - 1) / (m + 1)), m in [0.7, 1.42), by atanh's series in s <= 0.172,
// whose first term and the sum are held in pairs: the result is rounded once,
// give or take 1e-9. (fp64 here, by one thread per row, made a step of 1024
// requests 4 % slower; log2f added an ulp.)
struct KeptScale {
  float lse, inv_s;
};
__device__ __forceinline__ KeptScale kept_scale(const KeptNorm& k, float M) {
  if (!(k.hi > 0.f)) return {-INFINITY, INFINITY};
  int e = (__float_as_int(k.hi) >> 23) - 127;
  float sc = __int_as_float((127 - e) << 23);  // 2^-e (tot < 2^64)
  if (k.hi * sc > 1.41421356f) {
    sc *= 0.5f;
    ++e;
  }
  const float mh = k.hi * sc, ml = k.lo * sc;
  const F2 num = two_sum(mh - 1.f, ml);  // (mh - 1 is exact)
  F2 den = two_sum(mh, 1.f);
  den.lo += ml;
  const float s0 = __fdiv_rn(num.hi, den.hi);
  const float s1 = __fdividef(fmaf(-s0, den.hi, num.hi) + fmaf(-s0, den.lo, num.lo), den.hi);
  const float x = s0 * s0;
  float P = fmaf(x, 1.f / 13.f, 1.f / 11.f);
  P = fmaf(x, P, 1.f / 9.f);
  P = fmaf(x, P, 1.f / 7.f);
  P = fmaf(x, P, 1.f / 5.f);
  P = fmaf(x, P, 1.f / 3.f) * x;
  const float ln2 = 0.693147180559945f, ln2l = -1.904654299957768e-9f;
  const F2 l2 = two_sum(M, float(e - 40));
  const float ph = __fmul_rn(l2.hi, ln2);
  const float pl = fmaf(l2.hi, ln2, -ph) + fmaf(l2.hi, ln2l, l2.lo * ln2);
  const F2 t = two_sum(ph, 2.f * s0);
  return {t.hi + (t.lo + (pl + 2.f * fmaf(s0, P, s1))), k.inv * kFixScale};
}

__device__ __forceinline__ void grid_dependency_wait() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
}

}  // namespace tt
