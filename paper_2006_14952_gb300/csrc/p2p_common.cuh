// Helpers shared by the P2P kernels (one-sided p2p.cu, mutual p2p_mutual.cu):
// packed FP32x2 operand pairs, the one-instruction MUFU rsqrt, reciprocal and exp2,
// and the pair law with its constants as kernel parameters.
#pragma once

#include "common.cuh"

namespace hfmm {
namespace {

__device__ __forceinline__ float2 f2(float a) { return make_float2(a, a); }

// One MUFU instruction each (relative error about 2^-22); the arguments here are
// never denormal: r^2 > 0 in the cut-off range, and the exponent is -r^2 log2(e) / 4r_s^2 >= -7.3.
__device__ __forceinline__ float rsqrt_mufu(float x) {
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float rcp_mufu(float x) {
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float exp2_mufu(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// The pair-factor constants duplicated into (x, x) pairs, the operand form of the
// packed FP32x2 instructions, passed as kernel parameters (no register pairs to fill).
struct PairFit2 {
  float2 c[5];
  float2 a, p, kexp;  // see PairFit
  float2 pc0, pc1;    // polynomial split: -5 / (2 R_c^3), 3 / (2 R_c^5)
  float rc2;
};

// The host side of PairFit2 for a context.
inline PairFit2 pair_fit2(const Ctx &c) {
  PairFit2 f;
  auto two = [](float x) { return make_float2(x, x); };
  for (int j = 0; j < 5; ++j) f.c[j] = two(c.fit.c[j]);
  f.a = two(c.fit.a);
  f.p = two(c.fit.p);
  f.kexp = two(c.fit.kexp);
  f.pc0 = two((float)(-2.5 / (c.rc * c.rc * c.rc)));
  f.pc1 = two((float)(1.5 / (c.rc * c.rc * c.rc * c.rc * c.rc)));
  f.rc2 = c.fit.rc2;
  return f;
}

// r^2 of two pairs, less 2^-126: a pair at r = 0 comes out negative, so that one unsigned
// comparison of the bits takes 0 < r^2 < R_c^2 (a negative or a NaN is above every positive
// number): two instructions fewer of some 34 for two pairs, 2M P2P 7.97 -> 7.72 ms.
// Any r^2 of 2^-102 or more is unchanged; below that 1 / r^3 is beyond FP32.
__device__ __forceinline__ float2 pair_r2(float2 dx, float2 dy, float2 dz) {
  return __ffma2_rn(dx, dx, __ffma2_rn(dy, dy, __ffma2_rn(dz, dz, f2(-1.17549435e-38f))));
}
__device__ __forceinline__ bool in_cutoff(float r2, const PairFit2 &fit) {
  return __float_as_uint(r2) < __float_as_uint(fit.rc2);
}

// -f_(1)(r) of two pairs from their r^2.  kSplit 0: S(x) / r^3 = exp2(r^2 kexp)
// (P(v) / r + a) / r^2, 11 packed operations and a reciprocal (16 with a degree-9
// polynomial in r and 1/r^3 by itself: 8.57 -> 7.97 ms of P2P on the 2M set, k-d
// tree 16.3 -> 14.2; issue, FMA pipe and MUFU are now at 67, 53 and 49%.  One
// reciprocal for two pairs, 1/a = b / (a b): 8.26); 1: the polynomial truncation, 1/r^3 - 5 / (2 R_c^3) +
// 3 r^2 / (2 R_c^5).  Outside (0, R_c) the result may be inf or NaN.
template <int kSplit>
__device__ __forceinline__ float2 pair_factor2(float2 r2, const PairFit2 &fit) {
  const float2 ri = make_float2(rsqrt_mufu(r2.x), rsqrt_mufu(r2.y));
  const float2 ri2 = __fmul2_rn(ri, ri);
  if constexpr (kSplit == 1) {
    return __fadd2_rn(__fmul2_rn(ri2, ri), __ffma2_rn(r2, fit.pc1, fit.pc0));
  } else {
    const float2 d = __fadd2_rn(ri, fit.p);
    const float2 v = make_float2(rcp_mufu(d.x), rcp_mufu(d.y));
    float2 q = fit.c[4];
#pragma unroll
    for (int k = 3; k >= 0; --k) q = __ffma2_rn(q, v, fit.c[k]);
    const float2 g = __ffma2_rn(ri, q, fit.a);  // Q(x) / r
    const float2 e = __fmul2_rn(r2, fit.kexp);
    return __fmul2_rn(__fmul2_rn(make_float2(exp2_mufu(e.x), exp2_mufu(e.y)), g), ri2);
  }
}

}  // namespace
}  // namespace hfmm
