// Double-float arithmetic: a value is the unevaluated sum h + l of two FP32 numbers
// (about 48 significand bits), computed on the FP32 pipe with the error-free
// transformations of Dekker and Knuth (TwoSum, FastTwoSum, and the exact product
// a b = p + e with p = fl(a b), e = fma(a, b, -p)).  Sums and products are the
// "sloppy" double-float forms (relative error a few times 2^-48), enough for the
// FP64-accurate transforms of CMBWS_FP32X2.  Conversions from and to double run on
// the FP64 pipe and are kept out of inner loops.
#pragma once

#include <cuda_runtime.h>

namespace cmbws {

struct df {
  float h, l;
  df() = default;
  __host__ __device__ constexpr df(float h_, float l_) : h(h_), l(l_) {}
  __device__ df(double v) : h((float)v), l((float)(v - (double)(float)v)) {}
  __device__ explicit operator double() const { return (double)h + (double)l; }
};

__device__ __forceinline__ df two_sum(float a, float b) {
  const float s = a + b;
  const float bb = s - a;
  const float e = (a - (s - bb)) + (b - bb);
  return {s, e};
}
__device__ __forceinline__ df quick_two_sum(float a, float b) {
  const float s = a + b;
  return {s, b - (s - a)};
}
__device__ __forceinline__ df df_from(double v) { return df(v); }
__device__ __forceinline__ double df_to(df a) { return (double)a; }
__device__ __forceinline__ df df_mul(df a, df b) {
  const float p = a.h * b.h;
  float e = fmaf(a.h, b.h, -p);
  e = fmaf(a.h, b.l, e);
  e = fmaf(a.l, b.h, e);
  return quick_two_sum(p, e);
}
__device__ __forceinline__ df df_add(df a, df b) {
  const df s = two_sum(a.h, b.h);
  return quick_two_sum(s.h, s.l + (a.l + b.l));
}
__device__ __forceinline__ df df_sub(df a, df b) {
  const df s = two_sum(a.h, -b.h);
  return quick_two_sum(s.h, s.l + (a.l - b.l));
}
// a * b - c
__device__ __forceinline__ df df_fms(df a, df b, df c) {
  const float p = a.h * b.h;
  float e = fmaf(a.h, b.h, -p);
  e = fmaf(a.h, b.l, e);
  e = fmaf(a.l, b.h, e);
  const df s = two_sum(p, -c.h);
  return quick_two_sum(s.h, s.l + (e - c.l));
}
// Two FP32 values in one register pair: add.f32x2 and its kin round each half as the scalar
// instructions do.  They run at the scalar rate (2.2 cycles per warp for two additions against 1.15
// for one) but take one issue slot for both, which leaves the other one to loads and address work.
typedef unsigned long long f2;
__device__ __forceinline__ f2 f2_pack(float a, float b) {
  f2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ float2 f2_unpack(f2 v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}
__device__ __forceinline__ f2 f2_add(f2 a, f2 b) {
  f2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f2 f2_sub(f2 a, f2 b) {
  f2 r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f2 f2_mul(f2 a, f2 b) {
  f2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f2 f2_fma(f2 a, f2 b, f2 c) {
  f2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
// a factor of both halves in dot2_acc2: its words, and the upper one negated
struct dff {
  f2 h, l, nh;
  __device__ __forceinline__ explicit dff(df a) : h(f2_pack(a.h, a.h)), l(f2_pack(a.l, a.l)), nh(f2_pack(-a.h, -a.h)) {}
};
// Compensated accumulation acc_h + acc_l += a b of two sums (Dot2 of Ogita, Rump and Oishi 2005): a
// times the pair b.  The product is held negated, so that every step is an addition or a subtraction.
__device__ __forceinline__ void dot2_acc2(f2& acc_h, f2& acc_l, const dff& a, f2 bh, f2 bl) {
  const f2 np = f2_mul(a.nh, bh);
  f2 e = f2_fma(a.h, bh, np);
  e = f2_fma(a.h, bl, e);
  e = f2_fma(a.l, bh, e);
  const f2 s = f2_sub(acc_h, np);
  const f2 bb = f2_sub(s, acc_h);
  const f2 err = f2_sub(f2_sub(acc_h, f2_sub(s, bb)), f2_add(np, bb));
  acc_h = s;
  acc_l = f2_add(acc_l, f2_add(err, e));
}
// the rescaled Legendre recurrence step (A - A y) m1 - m2
__device__ __forceinline__ df df_recur(df A, df y, df m1, df m2) {
  const df ax = df_sub(A, df_mul(A, y));
  return df_fms(ax, m1, m2);
}

__device__ __forceinline__ df operator+(df a, df b) { return df_add(a, b); }
__device__ __forceinline__ df operator-(df a, df b) { return df_sub(a, b); }
__device__ __forceinline__ df operator*(df a, df b) { return df_mul(a, b); }
__device__ __forceinline__ df operator-(df a) { return {-a.h, -a.l}; }
__device__ __forceinline__ df& operator+=(df& a, df b) { return a = df_add(a, b); }
__device__ __forceinline__ df& operator-=(df& a, df b) { return a = df_sub(a, b); }
__device__ __forceinline__ df& operator*=(df& a, df b) { return a = df_mul(a, b); }

// complex double-float (16 bytes, the size of double2)
struct __align__(16) df2 {
  df x, y;
};

}  // namespace cmbws
