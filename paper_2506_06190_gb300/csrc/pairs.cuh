// Paired FP32 (sm_100 f32x2 instructions: one operation on both halves of a 64-bit register) and
// the phase reduction shared by the kernels that evaluate e^{ikr} over quadrature points.
#pragma once

#include <cuda_runtime.h>

namespace natbem {
namespace {

typedef unsigned long long u64;
__device__ __forceinline__ u64 pk(float lo, float hi) {
  u64 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ void upk(u64 v, float& lo, float& hi) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ u64 add2(u64 a, u64 b) {
  u64 d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ u64 sub2(u64 a, u64 b) {
  u64 d;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ u64 mul2(u64 a, u64 b) {
  u64 d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ u64 fma2(u64 a, u64 b, u64 c) {
  u64 d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ u64 bc(float x) { return pk(x, x); }

// 2 pi split for Cody-Waite reduction (Cody & Waite 1980): hi = 2 pi rounded to float,
// lo = float(2 pi - hi); rho - n hi - n lo with n = rint(rho / 2 pi) keeps |t| <= pi. Where an element's
// points share the centroid's n, |t| <= pi + k h for points within h of it. __sincosf is off by at
// most 4.0e-7 up to pi, 5e-7 at the k h of one that six elements a wavelength allow, 7e-7 at 2 pi and
// about |t| 2^-23 beyond (measured).
constexpr float kTwoPiHi = 6.28318548202514648f;
constexpr float kTwoPiLo = -1.7484555314695172e-7f;
constexpr float kInvTwoPi = 0.159154943091895336f;
// x + kRound - kRound rounds |x| < 2^22 to the nearest integer on the FMA pipe; the round
// instruction shares the quarter-rate unit with rsqrt, sin and cos.
constexpr float kRound = 12582912.f;

__device__ __forceinline__ u64 rsqrt2(u64 v) {
  float a, b;
  upk(v, a, b);
  return pk(rsqrtf(a), rsqrtf(b));
}
// nearest integers of rho / 2 pi
__device__ __forceinline__ u64 turns2(u64 rho) {
  return sub2(fma2(rho, bc(kInvTwoPi), bc(kRound)), bc(kRound));
}
// cos and sin of rho, n its turns or those of a nearby phase
__device__ __forceinline__ void sincos2(u64 rho, u64 n, u64& c, u64& s) {
  const u64 th = fma2(n, bc(-kTwoPiLo), fma2(n, bc(-kTwoPiHi), rho));
  float a, b, sa, ca, sb, cb;
  upk(th, a, b);
  __sincosf(a, &sa, &ca);
  __sincosf(b, &sb, &cb);
  c = pk(ca, cb);
  s = pk(sa, sb);
}

// The 7-point rule's outer points lie on the lines from the centroid to the vertices v_m: the
// first orbit (a, a, 1 - 2a) at (1 - 3a) v_m, the second at (1 - 3b) v_m, a, b = (6 -+ sqrt 15)/21.
// kOrbit is (1 - 3b) / (1 - 3a): a projection on a first-orbit offset gives the second's.
constexpr float kOrbit = -0.58957380768465f;

}  // namespace
}  // namespace natbem
