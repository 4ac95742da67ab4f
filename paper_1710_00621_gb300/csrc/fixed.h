// Fixed-point arithmetic of the FP64 Legendre stage (legendre_fx.cu).
//
// GB300 issues 1.9 FP64 multiply-adds per clock and SM, so the recurrence runs in 64-bit
// integers (a 32 x 32 -> 64 bit multiply issues at 56 per clock and SM) and the contraction on
// the FP16 tensor cores over 8-bit digits, whose products and sums are exact in FP32.
//
// Values.  mu_l (common.h: the rescaled Legendre values) is held as V = sigma mu 2^S, |V| < 2^62,
// with S = 62 - b chosen per m and ring pair from the largest |mu_l| up to the band-limit (|mu| < 2^b,
// recorded when the grid is planned; b is at most 4, and negative near the poles, where all values of a
// high m are small).  The sign sigma
// = + + - - by l - m modulo 4 turns mu_l = A x mu_{l-1} - mu_{l-2} into V2 - A x V1 (l - m even) and
// V2 + A x V1 (odd); the coefficients (synthesis) or the results (adjoint) take sigma back.
// For the products V = h 2^32 + l with both words signed: the state holds V + 2^31, whose upper word
// is h and whose lower one is l + 2^31.  For the contraction the bytes of V + 2^63 are its base-256
// digits, byte 7 less 128, the others as they are.
// Before a pair's values are near their largest (they grow from where its walk starts; smaller ones have
// no digits), V carries a binary exponent e (a multiple of 8): mu = V 2^-(S + e), V shifted down by 8
// bits as it grows; e is 0 from 2^-7 of the largest on.
//
// Coefficients a (synthesis) and ring parts times 2^-S of their pair (adjoint) are scaled by a power of
// two per (m, map) to |a| < 2^62 and split
// into 8 signed digits (-128..127).  With digits u_i of V (8 of them, from byte 7 down) and d_j of a,
// the contraction sums u_i d_j for i + j <= 7 in FP32: u is passed as an FP16 subnormal (the byte
// itself, u 2^-24), d as an FP16 integer; |sum| < 2^24 units over 64 terms of 8 products each, so
// every sum is exact (slices with exact sums: Ozaki, Ogita, Oishi and Rump 2012).  The dropped products
// are 2^-61 of the largest one.  With 7 digits of each (2^-55) a spectrum falling as l^-3 came out 2 to 4
// times less accurate than from FP64 arithmetic, a monopole and dipole under L = 767 three times; the eighth
// costs 3 to 4 % (Nside 1024, 3 maps: 20.9 -> 21.6 ms).  Integer sums do not depend on their order
// or on the tile.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <climits>

namespace cmbws {

typedef long long fx_t;
typedef unsigned long long fxu_t;

constexpr int kFxABits = 62;  // coefficients and ring parts: |a| < 2^62
constexpr fx_t kFxBias = 1ll << 31;
constexpr int kFxDig = 8;     // digits of both factors
constexpr int kFxBlk = 8;     // sums kept: i + j = 0..7

// 32 x 32 -> 64 bit products as PTX: with C expressions in their place the synthesis of 3 maps at Nside
// 1024 takes 25.7 ms instead of 21.9, the adjoint of a map at GL L = 1000 917 us instead of 802.
__device__ __forceinline__ fx_t fx_mul(int a, int b) {
  fx_t r;
  asm("mul.wide.s32 %0, %1, %2;" : "=l"(r) : "r"(a), "r"(b));
  return r;
}
__device__ __forceinline__ fxu_t fx_mulu(unsigned a, unsigned b) {
  fxu_t r;
  asm("mul.wide.u32 %0, %1, %2;" : "=l"(r) : "r"(a), "r"(b));
  return r;
}

// S from the high word of the largest |mu|
__device__ __forceinline__ int fx_scale(unsigned mu_hi) { return 62 - ((int)(mu_hi >> 20) - 1022); }

// v 2^k rounded to nearest (v finite, |v 2^k| < 2^63)
__device__ __forceinline__ fx_t fx_from_double(double v, int k) {
  const fxu_t b = (fxu_t)__double_as_longlong(v);
  const int be = (int)((b >> 52) & 0x7ff);
  const fxu_t m = (b & 0xfffffffffffffull) | (be ? 1ull << 52 : 0ull);
  const int s = max(be, 1) - 1075 + k;  // v = m 2^(max(be, 1) - 1075)
  fxu_t r;
  if (s >= 0) r = s < 64 ? m << s : 0;
  else r = s > -64 ? (m + (1ull << (-s - 1))) >> -s : 0;
  return (b >> 63) ? -(fx_t)r : (fx_t)r;
}
// Digits of two scaled coefficients as FP16 integers, the first in the lower half: w[j] holds the
// digits d_j (j = 0 the leading one).  1024 + u has a byte u in its lowest mantissa bits; minus
// 1152 leaves u - 128 exactly.
__device__ __forceinline__ void fx_coef_digits(fx_t v0, fx_t v1, unsigned (&w)[kFxDig]) {
  const fxu_t a = (fxu_t)v0 + 0x8080808080808080ull, b = (fxu_t)v1 + 0x8080808080808080ull;
#pragma unroll
  for (int j = 0; j < kFxDig; ++j) {
    const int byte = kFxDig - 1 - j;
    const unsigned x = (unsigned)(byte < 4 ? a : a >> 32), y = (unsigned)(byte < 4 ? b : b >> 32);
    const unsigned sel = (unsigned)(byte & 3);
    unsigned t = __byte_perm(x, y, sel | ((sel + 4) << 4));       // bytes u0, u1
    t = __byte_perm(t, 0x64646464u, 0x4140);                      // 0x64 above each
    asm("sub.rn.f16x2 %0, %1, %2;" : "=r"(w[j]) : "r"(t), "r"(0x64806480u));
  }
}

// A_lm as {upper word, signed lower word, shift, rounding constant} of a recurrence step: with
// A < 2^sh the words hold A 2^(62 - sh), the shift is 3 + sh
__device__ __forceinline__ int4 fx_coef(double A) {
  if (!(A > 0.0)) return make_int4(0, 0, 3, 0);
  const fxu_t b = (fxu_t)__double_as_longlong(A);
  const int E = (int)((b >> 52) & 0x7ff) - 1023;
  const int sh = max(E + 1, 0);
  const fxu_t m = ((b & 0xfffffffffffffull) | (1ull << 52)) << (10 + E - sh);  // E >= -10
  return make_int4((int)((m + (1ull << 31)) >> 32), (int)m, 3 + sh, 1 << (28 - sh));
}

// A x V1 rounded; V1 is biased, x = xh 2^32 + xl holds cos(theta) 2^63.  A x is formed as
// A x 2^(61 - sh) plus 2^31, so that its words split as V's do (the lower word of A is signed: the sum
// of the three lower terms then fits 32 bits).  The parts dropped from it are one unit on average,
// which is put back: a constant error of A x is a drift of the phase.  The product with V1 keeps 96
// bits of which the shift takes the upper 64 (dropped: below 2 units).
// With biased words and sums of signed products a step takes 42 issue cycles per warp; with the words
// split from an unbiased V and the cross products summed as unsigned it took 47.
__device__ __forceinline__ fx_t fx_ax(int4 A, unsigned xh, unsigned xl, fx_t V1) {
  const unsigned u = (unsigned)(fx_mulu((unsigned)A.x, xl) >> 32) + (unsigned)((fxu_t)fx_mul(A.y, (int)xh) >> 32) +
                     0x80000001u;
  const fxu_t X = fx_mulu((unsigned)A.x, xh) + u;
  const int Xl = (int)((unsigned)X - 0x80000000u), Xh = (int)(X >> 32);
  const int Vl = (int)((unsigned)V1 - 0x80000000u), Vh = (int)((fxu_t)V1 >> 32);
  const fx_t cr = fx_mul(Xl, Vh) + fx_mul(Xh, Vl) + (fx_t)(unsigned)A.w;
  const fx_t hh = fx_mul(Xh, Vh) + (fx_t)(int)(cr >> 32);
  const unsigned lo = (unsigned)hh, hi = (unsigned)((fxu_t)hh >> 32);
  const unsigned ph = __funnelshift_l(lo, hi, A.z), pl = __funnelshift_l((unsigned)cr, lo, A.z);
  return (fx_t)(((fxu_t)ph << 32) | pl);
}

// Row state of one ring pair: the last two values (V1 at l - 1, V2 at l - 2), biased, and their
// exponent.  A pair that has not started holds zeros.
struct FxState {
  fx_t V1 = kFxBias, V2 = kFxBias;
  int e = 0;
  // two steps, l - m even and l + 1; the new values are V2 and V1
  __device__ __forceinline__ void step2(int4 A0, int4 A1, unsigned xh, unsigned xl) {
    const fx_t a = V2 - fx_ax(A0, xh, xl, V1);
    V2 = a;
    V1 += fx_ax(A1, xh, xl, a);
  }
};

// values (mu_l, mu_l+1), l - m even, sigma of l +, at scale S -> state whose V2, V1 are those two values
__device__ __forceinline__ FxState fx_start(double v0, double v1, int S) {
  FxState st;
  const unsigned h = max((unsigned)__double2hiint(v0) & 0x7fffffffu,
                         (unsigned)__double2hiint(v1) & 0x7fffffffu);
  if (h == 0) return st;
  // |V| < 2^(S + e + E), E = exponent bound of the larger value: at most 2^59 unless e is 0 (walks start
  // from |V| = 2 at e = 0 on, so e is at most 56)
  st.e = max(0, 59 - S - ((int)(h >> 20) - 1022)) & ~7;
  st.V2 = fx_from_double(v0, S + st.e) + kFxBias;
  st.V1 = fx_from_double(v1, S + st.e) + kFxBias;
  return st;
}

// The state at a checkpoint in two words: values shifted up by one bit, or by four over the exponent
// (bit 0 set, bits 1-3 its eighths less one; such values are below 2^59).  Two shifts bring them back;
// converting FP64 checkpoints at every use, and the adjoint's ring parts in every tile of l, took a tenth
// of the adjoint (Nside 1024, 3 maps: 20.4 -> 18.2 ms).
__device__ __forceinline__ ulonglong2 fx_pack(double v0, double v1, int S) {
  const FxState st = fx_start(v0, v1, S);
  const fxu_t a = (fxu_t)(st.V2 - kFxBias), b = (fxu_t)(st.V1 - kFxBias);
  if (st.e == 0) return make_ulonglong2(a << 1, b << 1);
  return make_ulonglong2(a << 4 | (fxu_t)(2 * (st.e / 8 - 1) + 1), b << 4);
}
__device__ __forceinline__ FxState fx_unpack(ulonglong2 c) {
  FxState st;
  int sh = 1;
  if (c.x & 1) {
    st.e = 8 * ((int)((c.x >> 1) & 7) + 1);
    sh = 4;
  }
  st.V2 = ((fx_t)c.x >> sh) + kFxBias;
  st.V1 = ((fx_t)c.y >> sh) + kFxBias;
  return st;
}

// sigma of l -
__device__ __forceinline__ void fx_negate(FxState& st) {
  st.V2 = 2 * kFxBias - st.V2;
  st.V1 = 2 * kFxBias - st.V1;
}

// room for a step with coefficient A while an exponent is left: |V| below 2^(61 - sh)
__device__ __forceinline__ void fx_renorm(FxState& st, int4 A) {
  const int ah = (int)(st.V1 >> 32), bh = (int)(st.V2 >> 32);
  const int h = max(ah ^ (ah >> 31), bh ^ (bh >> 31));
  if (st.e > 0 && (h >> (32 - A.z)) != 0) {
    st.V1 = ((st.V1 - kFxBias + 128) >> 8) + kFxBias;
    st.V2 = ((st.V2 - kFxBias + 128) >> 8) + kFxBias;
    st.e -= 8;
  }
}

// the value V (biased) at exponent e brought to exponent 0
__device__ __forceinline__ fx_t fx_emit(fx_t V, int e) {
  if (e == 0) return V;
  return (e > 62 ? 0 : (V - kFxBias + (1ll << (e - 1))) >> e) + kFxBias;
}

// step2 of a pair that may start at l (with the state s0) or still carry an exponent
__device__ __forceinline__ void fx_step2_slow(FxState& st, int4 A0, int4 A1, unsigned xh, unsigned xl,
                                              bool start, const FxState& s0) {
  fx_renorm(st, A0);
  st.V2 -= fx_ax(A0, xh, xl, st.V1);
  fx_renorm(st, A1);
  st.V1 += fx_ax(A1, xh, xl, st.V2);
  if (start) st = s0;
}

// Digits of biased values as FP16 subnormals: the bytes of V + 2^63.  fx_bytes adds what the state lacks
// of that; fx_digits2 turns 16 bits (word w, upper half if HI) of two consecutive values (the first in the
// lower halves of the results) into two digit words, the leading digit in d0.
__device__ __forceinline__ fxu_t fx_bytes(fx_t V) { return (fxu_t)V + ((1ull << 63) - (fxu_t)kFxBias); }
template <int Q>  // bits 16 Q..16 Q + 15: digits 6 - 2 Q (d0) and 7 - 2 Q (d1)
__device__ __forceinline__ void fx_digits2(fxu_t a, fxu_t b, unsigned& d0, unsigned& d1) {
  const unsigned x = (unsigned)(Q < 2 ? a : a >> 32), y = (unsigned)(Q < 2 ? b : b >> 32);
  const unsigned p = __byte_perm(x, y, (Q & 1) ? 0x7632 : 0x5410);
  d0 = __byte_perm(p, 0, 0x4341);
  d1 = p & 0x00ff00ffu;
}

// Sums of one output column: sum_s I_s 2^(8 (7 - s)) over the blocks s = i + j, kept as
// H 2^32 + L (H the blocks 0..3).
struct FxSum {
  fx_t H = 0, L = 0;
  // I_s of one drain; |I_s| < 2^24, and I_0, I_2 (fewer products, smaller leading digits) below
  // 2^23, so that the upper blocks combine pairwise in 32 bits
  __device__ __forceinline__ void add(int s, int v, int& prev) {
    if (s == 0 || s == 2) prev = v;
    else if (s == 1) H += fx_mul(prev * 256 + v, 65536);
    else if (s == 3) H += (fx_t)(prev * 256 + v);
    else if (s < 7) L += fx_mul(v, 1 << (8 * (7 - s)));
    else L += (fx_t)v;
  }
  // less 128 times the sum of the coefficients (sum, 2^-30 of it in hi), for byte 7 stored plus
  // 128: 128 sum_k a_k in these units
  __device__ __forceinline__ double value(fx_t shi, fx_t slo, int k) const {
    const fx_t h = H - (shi << 5), l = L - (slo << 7);
    return scalbn((double)h * 4294967296.0 + (double)l, k);
  }
};

}  // namespace cmbws
