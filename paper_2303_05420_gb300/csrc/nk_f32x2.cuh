// Packed FP32 arithmetic (two FP32 values in one 64-bit register pair) and
// the activation maps over it.
//
// sm_103a executes add / mul / fma on f32x2 at the FP32 rate of the scalar
// instructions (measured: 120.7 lane-FMAs per SM and cycle packed, 115.6
// scalar) but from half the issue slots, so kernels that are bound by
// instruction issue rather than by the FP32 pipe gain (measured: 16 scalar
// FMAs beside 8 shift-and-xor pairs 3.04 ms, 8 packed FMAs beside the same
// 2.13 ms).  Each half rounds as the scalar instruction does.
#pragma once

#include "nk_map.cuh"

struct f2 {
  unsigned long long u;
};

__device__ __forceinline__ f2 f2_make(float lo, float hi) {
  f2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r.u) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ f2 f2_dup(float x) { return f2_make(x, x); }
__device__ __forceinline__ float f2_lo(f2 a) {
  float x;
  asm("{\n\t.reg .f32 t;\n\tmov.b64 {%0, t}, %1;\n\t}" : "=f"(x) : "l"(a.u));
  return x;
}
__device__ __forceinline__ float f2_hi(f2 a) {
  float x;
  asm("{\n\t.reg .f32 t;\n\tmov.b64 {t, %0}, %1;\n\t}" : "=f"(x) : "l"(a.u));
  return x;
}
__device__ __forceinline__ f2 f2_fma(f2 a, f2 b, f2 c) {
  f2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.u) : "l"(a.u), "l"(b.u), "l"(c.u));
  return r;
}
__device__ __forceinline__ f2 f2_mul(f2 a, f2 b) {
  f2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.u) : "l"(a.u), "l"(b.u));
  return r;
}
// a b clamped to [0, 1] (0 for a NaN): the clamp is the scalar
// multiplication's own, which the packed one has not.
__device__ __forceinline__ f2 f2_mul_sat(f2 a, f2 b) {
  return f2_make(__saturatef(f2_lo(a) * f2_lo(b)), __saturatef(f2_hi(a) * f2_hi(b)));
}
__device__ __forceinline__ f2 f2_add(f2 a, f2 b) {
  f2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.u) : "l"(a.u), "l"(b.u));
  return r;
}

__device__ __forceinline__ f2 f2_sub(f2 a, f2 b) {
  f2 r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r.u) : "l"(a.u), "l"(b.u));
  return r;
}

// nk_B_poly / pi on both halves: the maps below give J / pi = c + (1 -
// c)^{3/2} B(c) / pi, one multiplication fewer than J, with pi in the layers'
// folded factor (relative error of J / pi with these FP32 coefficients 4.0e-8;
// nk_J01_f32's constants give 4.9e-8).
//
// DEEP: a fit with next to no mean error (4.3e-8 at c = 0, 1e-8 from c = 0.3 on;
// csrc/fit_jpos.py pi), for the Flatten readout of many layers without a pool,
// where errors of one sign add up: 2.4e-8 (rms, eight layers of 32x32, 300 x 250
// images) against 3.7e-8 with the other one and a rounded layer constant.  The
// pooled nets are closer with the other one, which their folded factors' rounding
// offsets (Myrtle-10, 50 x 63: 2.8e-8, and 3.1e-8 with this one).
template <bool DEEP = false>
__device__ __forceinline__ f2 nk_Bpi_poly2(f2 c) {
  f2 p = f2_dup(DEEP ? -2.113373776e-04f : -2.236311266e-04f);
  p = f2_fma(p, c, f2_dup(DEEP ? 9.120404720e-04f : 9.384872974e-04f));
  p = f2_fma(p, c, f2_dup(DEEP ? -2.336561447e-03f : -2.355845412e-03f));
  p = f2_fma(p, c, f2_dup(DEEP ? 5.963813979e-03f : 5.969292484e-03f));
  p = f2_fma(p, c, f2_dup(DEEP ? -2.253376879e-02f : -2.253424563e-02f));
  p = f2_fma(p, c, f2_dup(3.183098733e-01f));
  return p;
}

// u sqrt(u) on both halves, u >= 0.
__device__ __forceinline__ f2 nk_u32(f2 u) {
  return f2_mul(u, f2_make(nk_sqrt_approx(f2_lo(u)), nk_sqrt_approx(f2_hi(u))));
}

// J(c) / pi for c in [0, 1] on both halves (nk_J01_f32).  The caller clamps
// (f2_mul_sat): c = K a a' is above 1 not only by rounding, and the polynomial
// has no bound there.  Where sqrt(q q') < 2.9e-39 the product a a' of the
// factors 1 / sqrt(q) is infinite, c infinite or (K = 0) a NaN, and such a
// pixel pair, which adds b b' J ~ 1e-39, would spoil the whole entry.
template <bool DEEP = false>
__device__ __forceinline__ f2 nk_Jpi01_2(f2 c) {
  return f2_fma(nk_u32(f2_sub(f2_dup(1.f), c)), nk_Bpi_poly2<DEEP>(c), c);
}

// J(c) / pi for any c on both halves (nk_J_f32; c beyond [-1, 1] counts as the
// nearer end, a NaN gives 0): J(|c|) + pi min(c, 0) = pi max(c, 0) + (1 -
// |c|)^{3/2} B(|c|).
template <bool DEEP = false>
__device__ __forceinline__ f2 nk_Jpi_2(f2 c) {
  const float c0 = f2_lo(c), c1 = f2_hi(c);
  const f2 a = f2_make(fminf(fabsf(c0), 1.f), fminf(fabsf(c1), 1.f));
  return f2_fma(nk_u32(f2_sub(f2_dup(1.f), a)), nk_Bpi_poly2<DEEP>(a), f2_make(__saturatef(c0), __saturatef(c1)));
}

// asin(c) for c in [-1, 1] (nk_asin_f32; values outside by rounding act as
// +-1) on both halves, and sqrt(1 - c^2).
__device__ __forceinline__ f2 nk_asin_sqrt_2(f2 c, f2* sn) {
  const float c0 = f2_lo(c), c1 = f2_hi(c);
  const f2 om = f2_fma(f2_mul(c, f2_dup(-1.f)), c, f2_dup(1.f));
  const float s0 = nk_sqrt_approx(fmaxf(f2_lo(om), 0.f)), s1 = nk_sqrt_approx(fmaxf(f2_hi(om), 0.f));
  const f2 m = f2_make(fminf(fabsf(c0), s0), fminf(fabsf(c1), s1));
  const f2 z = f2_mul(m, m);
  f2 p = f2_dup(1.112414098e-01f);
  p = f2_fma(p, z, f2_dup(-9.249696326e-02f));
  p = f2_fma(p, z, f2_dup(7.689475858e-02f));
  p = f2_fma(p, z, f2_dup(1.641334877e-02f));
  p = f2_fma(p, z, f2_dup(4.649848860e-02f));
  p = f2_fma(p, z, f2_dup(7.488511025e-02f));
  p = f2_fma(p, z, f2_dup(1.666690495e-01f));
  const f2 as = f2_fma(f2_mul(m, z), p, m);
  const f2 co = f2_sub(f2_dup(NK_HALF_PI_F), as);
  *sn = f2_make(s0, s1);
  return f2_make(copysignf(fabsf(c0) > s0 ? f2_lo(co) : f2_lo(as), c0),
                 copysignf(fabsf(c1) > s1 ? f2_hi(co) : f2_hi(as), c1));
}
__device__ __forceinline__ f2 nk_asin_2(f2 c) {
  f2 sn;
  return nk_asin_sqrt_2(c, &sn);
}
