// Ring FFT stage of FP64 transforms in 64-bit fixed point (block floating point) on the integer
// units: a complex multiply costs about 70 issue cycles per warp here against 270 on the FP64 pipe
// (1.9 multiply-adds per clock and SM), an addition 2.3 against 68.
//
// The transform of each ring pair, its plans, the shared-memory swizzle and the three modes are
// those of ringfft.cu.  Values are complex pairs of 64-bit integers with one power-of-two scale per
// ring pair, taken from the largest input (a scan before the transform), with modulus <= 2^61.
// * A pass of S radix-2 stages (register groups of 2^S) can grow values by 2^S.  Every pass records
//   the largest value that it stores, and the next one shifts its inputs down by the bits that are
//   missing (or up by those that are free), so the values stay near 2^61 whatever the spectrum.
// * A pass's position-dependent twiddles are applied at once, to element k the rev_S(k)-th power of
//   one root (7 multiplies for three stages instead of 12), and the stages then only need 8th roots
//   of unity.
// * Factors (twiddles, chirps, filters, phases) are fixed point with 61 fraction bits, as an upper
//   digit and a balanced lower one of 31 bits; a product keeps the three leading partial products
//   (dropped: below 2 units of the last place).
// The 1 / sqrt(2) and sqrt(2) of the m > 0 terms are applied by the Legendre stage (legendre_fx.cu).
// Rounding: a few units of the last place (2^-60 of the largest value) per pass; the factors are made from
// FP64 values, so they add 2^-54 of it per pass, as in FP64 arithmetic.
// Synthesis of 3 maps at Nside 1024: 6.3 ms on the FP64 pipe, 1.9 ms here; analysis of a map on a GL grid
// of L = 1000 570 -> 130 us.
#include "common.h"
#include "fixed.h"

namespace cmbws {

namespace {

struct __align__(16) cx {
  fx_t x, y;
};

__device__ __forceinline__ cx operator+(cx a, cx b) { return {a.x + b.x, a.y + b.y}; }
__device__ __forceinline__ cx operator-(cx a, cx b) { return {a.x - b.x, a.y - b.y}; }
// a + v, or a - v; modulo 2^64
__device__ __forceinline__ cx wrap_add(cx a, cx v, bool neg) {
  const fxu_t x = (fxu_t)v.x, y = (fxu_t)v.y;
  return {(fx_t)((fxu_t)a.x + (neg ? 0 - x : x)), (fx_t)((fxu_t)a.y + (neg ? 0 - y : y))};
}
__device__ __forceinline__ cx cconj(cx a) { return {a.x, -a.y}; }

// digits of a value: v = h 2^32 + 2 l (its last bit dropped), l >= 0
__device__ __forceinline__ int dig_h(fx_t v) { return (int)(v >> 32); }
__device__ __forceinline__ int dig_l(fx_t v) { return (int)((unsigned)v >> 1); }
// (2^61-scaled product) hh 2^63 + cross 2^32, shifted back and rounded
__device__ __forceinline__ fx_t join(fx_t hh, fx_t cross) { return (hh << 2) + ((cross + (1 << 28)) >> 29); }

// a w, or a conj(w): w = {re upper, re lower, im upper, im lower}, digits of 31 bits
template <bool CONJ>
__device__ __forceinline__ cx cmul(cx a, int4 w) {
  const int xh = dig_h(a.x), xl = dig_l(a.x), yh = dig_h(a.y), yl = dig_l(a.y);
  const fx_t ph = fx_mul(xh, w.x), pc = fx_mul(xh, w.y) + fx_mul(xl, w.x);  // x re
  const fx_t qh = fx_mul(yh, w.z), qc = fx_mul(yh, w.w) + fx_mul(yl, w.z);  // y im
  const fx_t rh = fx_mul(xh, w.z), rc = fx_mul(xh, w.w) + fx_mul(xl, w.z);  // x im
  const fx_t sh = fx_mul(yh, w.x), sc = fx_mul(yh, w.y) + fx_mul(yl, w.x);  // y re
  return CONJ ? cx{join(ph + qh, pc + qc), join(sh - rh, sc - rc)}
              : cx{join(ph - qh, pc - qc), join(sh + rh, sc + rc)};
}
__device__ __forceinline__ fx_t rmul(fx_t v, int h, int l) {
  const int vh = dig_h(v);
  return join(fx_mul(vh, h), fx_mul(vh, l) + fx_mul(dig_l(v), h));
}
// times sqrt(1/2): sqrt(1/2) 2^61 = 759250125 2^31 - 12858224
__device__ __forceinline__ fx_t mul_rsqrt2(fx_t v) { return rmul(v, 759250125, -12858224); }

// v 2^-s rounded (s > 0), or v 2^-s (s <= 0)
__device__ __forceinline__ fx_t shift_down(fx_t v, int s) { return s > 0 ? (v + (1ll << (s - 1))) >> s : v << -s; }

// v 2^ex as double, rounded to nearest
__device__ __forceinline__ double fx_value(fx_t v, int ex) {
  const fxu_t u = (fxu_t)(v < 0 ? -v : v);
  if (u == 0) return 0.0;
  const int lz = __clzll((long long)u);
  const fxu_t m = u << lz;
  const int be = 1023 + 63 - lz + ex;  // biased exponent before rounding
  const fxu_t r = (m >> 11) + ((m >> 10) & 1);
  if (be < 1 || be > 2045) return scalbn((double)v, ex);
  return __longlong_as_double((long long)(((fxu_t)(be - 1) << 52) + r) | (v < 0 ? (long long)(1ull << 63) : 0ll));
}

// the transform buffer: the swizzle of ringfft.cu
struct Sbuf {
  cx* p;
  int sh;
  __device__ __forceinline__ cx& operator[](int i) const { return p[(i ^ ((i >> sh) & 15)) + (i >> 4)]; }
};

// x times exp(-2 pi i c / 2^e) (INV: the conjugate), e <= 3
template <bool INV>
__device__ __forceinline__ cx unit_mul(cx x, int c, int e) {
  const int q = (c << (3 - e)) & 3;  // eighths; c < 2^(e-1), so the angle is below pi
  if (q == 0) return x;
  if (q == 2) return INV ? cx{-x.y, x.x} : cx{x.y, -x.x};
  const fx_t a = mul_rsqrt2(x.x + x.y), b = mul_rsqrt2(x.x - x.y);
  // (x + i y)(1 - i) / sqrt2 = (x + y) - i (x - y); times -i once more for q = 3
  if (q == 1) return INV ? cx{b, a} : cx{a, -b};
  return INV ? cx{-a, b} : cx{-b, -a};
}

__host__ __device__ constexpr int rev_bits(int k, int S) {
  return S == 1 ? k : S == 2 ? ((k & 1) << 1) | (k >> 1) : ((k & 1) << 2) | (k & 2) | (k >> 2);
}

__device__ __forceinline__ unsigned hi_abs(fx_t v) {
  const int h = (int)(v >> 32);
  return (unsigned)(h ^ (h >> 31));
}
__device__ __forceinline__ unsigned hi_abs(cx v) { return max(hi_abs(v.x), hi_abs(v.y)); }

// Renormalisation between passes: the largest upper word of a pass's results (three slots in shared
// memory, rotating: one written, one read, one cleared) and the shift that follows from it.
struct Renorm {
  unsigned* slot;  // [3], zero before the first pass (a barrier in between)
  int pass = 0;
  int gain = 0;      // bits free above the last pass's results
  int shifted = 0;   // bits shifted down since the last reset
  __device__ __forceinline__ void begin() {
    if (threadIdx.x == 0) slot[(pass + 1) % 3] = 0;
  }
  // ends a pass (barrier) whose largest upper word in this thread is mx
  __device__ __forceinline__ void end(unsigned mx) {
    mx = __reduce_max_sync(0xffffffffu, mx);
    if ((threadIdx.x & 31) == 0) atomicMax(&slot[pass % 3], mx);
    __syncthreads();
    // components below 2^(64 - clz) -> below 2^60, modulus below 2^61
    const unsigned h = slot[pass % 3];
    gain = h ? __clz(h) - 4 : 0;
    ++pass;
  }
  // the shift of the next pass's inputs, S stages
  __device__ __forceinline__ int next(int S) {
    const int down = S - gain;
    shifted += down;
    return down;
  }
};

// tw[j] = exp(-2 pi i j / nmax), j < nmax.  mx: the largest upper word stored.  Decimation in time, S stages from s0 (1-based) on:
// bit-reversed in, natural out; down: the shift of the inputs.
template <int S, bool INV, typename LD, typename ST>
__device__ __forceinline__ void dit_group(Sbuf buf, int g, int s0, const int4* __restrict__ tw, int nmax,
                                          int down, bool first, bool last, const LD& ld, const ST& st,
                                          unsigned& mx) {
  constexpr int E = 1 << S;
  const int half0 = 1 << (s0 - 1);
  const int pos0 = g & (half0 - 1);
  const int base = ((g >> (s0 - 1)) << (s0 - 1 + S)) + pos0;
  const int step = pos0 * (nmax >> (s0 + S - 1));
  cx x[E];
#pragma unroll
  for (int k = 0; k < E; ++k) {
    const cx v = first ? ld(base + k * half0) : buf[base + k * half0];
    x[k] = {shift_down(v.x, down), shift_down(v.y, down)};
  }
  if (step != 0) {
#pragma unroll
    for (int k = 1; k < E; ++k) x[k] = cmul<INV>(x[k], tw[step * rev_bits(k, S)]);
  }
#pragma unroll
  for (int t = 0; t < S; ++t)
#pragma unroll
    for (int c = 0; c < (1 << t); ++c)
#pragma unroll
      for (int k0 = 0; k0 < E; k0 += 2 << t) {
        const int k = k0 + c;
        const cx v = unit_mul<INV>(x[k + (1 << t)], c, t + 1);
        x[k + (1 << t)] = x[k] - v;
        x[k] = x[k] + v;
      }
#pragma unroll
  for (int k = 0; k < E; ++k) {
    if (last) {
      st(base + k * half0, x[k]);
    } else {
      buf[base + k * half0] = x[k];
      mx = max(mx, hi_abs(x[k]));
    }
  }
}

// Decimation in frequency, S stages from s1 down: natural in, bit-reversed out (forward only).
template <int S, typename LD, typename ST>
__device__ __forceinline__ void dif_group(Sbuf buf, int g, int s1, const int4* __restrict__ tw, int nmax,
                                          int down, bool first, bool last, const LD& ld, const ST& st,
                                          unsigned& mx) {
  constexpr int E = 1 << S;
  const int h = 1 << (s1 - S);
  const int pos0 = g & (h - 1);
  const int base = ((g >> (s1 - S)) << s1) + pos0;
  const int step = pos0 * (nmax >> s1);
  cx x[E];
#pragma unroll
  for (int k = 0; k < E; ++k) {
    const cx v = first ? ld(base + k * h) : buf[base + k * h];
    x[k] = {shift_down(v.x, down), shift_down(v.y, down)};
  }
#pragma unroll
  for (int t = 0; t < S; ++t) {
    const int sh = S - 1 - t;
#pragma unroll
    for (int c = 0; c < (1 << sh); ++c)
#pragma unroll
      for (int k0 = 0; k0 < E; k0 += 2 << sh) {
        const int k = k0 + c;
        const cx d = x[k] - x[k + (1 << sh)];
        x[k] = x[k] + x[k + (1 << sh)];
        x[k + (1 << sh)] = unit_mul<false>(d, c, sh + 1);
      }
  }
  if (step != 0) {
#pragma unroll
    for (int k = 1; k < E; ++k) x[k] = cmul<false>(x[k], tw[step * rev_bits(k, S)]);
  }
#pragma unroll
  for (int k = 0; k < E; ++k) {
    if (last) {
      st(base + k * h, x[k]);
    } else {
      buf[base + k * h] = x[k];
      mx = max(mx, hi_abs(x[k]));
    }
  }
}

// groups of 8 elements where every thread has one, of 4 where half of the threads have one, else of 2: a
// larger group saves passes and twiddles, but is one thread's serial work.  Rings of 127 pixels (length
// 256, 128 threads; 34 launches of a solve): 1107 us with groups of 2, 965 with groups of 4, 1248 with
// groups of 8; groups of 8 for half of the threads slow rings of 256 pixels and less by 3 %.
__device__ __forceinline__ int group_stages(int N) {
  const int nt = (int)blockDim.x;
  return (N >> 3) >= nt ? 3 : (N >> 1) >= nt ? 2 : 1;
}

// Transforms of size N.  The last pass's st(i, v) may record its own largest upper word in mx.
template <bool INV, typename LD, typename ST>
__device__ void fft_dit(Sbuf buf, int N, const int4* __restrict__ tw, int nmax, Renorm& rn, unsigned& mx,
                        const LD& ld, const ST& st) {
  const int S = group_stages(N);
  const int n = 31 - __clz(N);
  const int r = n % S, np = n == 0 ? 1 : n / S + (r ? 1 : 0);
  int s0 = 1;
  for (int pass = 0; pass < np; ++pass) {
    const bool first = pass == 0, last = pass == np - 1;
    const int st_ = n == 0 ? 0 : (pass < n / S) ? S : r;
    rn.begin();
    const int down = rn.next(st_);
    mx = 0;
    if (st_ == 3) {
      for (int g = threadIdx.x; g < (N >> 3); g += blockDim.x)
        dit_group<3, INV>(buf, g, s0, tw, nmax, down, first, last, ld, st, mx);
    } else if (st_ == 2) {
      for (int g = threadIdx.x; g < (N >> 2); g += blockDim.x)
        dit_group<2, INV>(buf, g, s0, tw, nmax, down, first, last, ld, st, mx);
    } else if (st_ == 1) {
      for (int g = threadIdx.x; g < (N >> 1); g += blockDim.x)
        dit_group<1, INV>(buf, g, s0, tw, nmax, down, first, last, ld, st, mx);
    } else if (threadIdx.x == 0) {  // one point
      const cx v = ld(0);
      st(0, cx{shift_down(v.x, down), shift_down(v.y, down)});
    }
    s0 += st_;
    rn.end(mx);
  }
}

template <typename LD, typename ST>
__device__ void fft_dif(Sbuf buf, int N, const int4* __restrict__ tw, int nmax, Renorm& rn, unsigned& mx,
                        const LD& ld, const ST& st) {
  const int S = group_stages(N);
  const int n = 31 - __clz(N);
  const int r = n % S, np = n == 0 ? 1 : n / S + (r ? 1 : 0);
  int s1 = n;
  for (int pass = 0; pass < np; ++pass) {
    const bool first = pass == 0, last = pass == np - 1;
    const int st_ = n == 0 ? 0 : (pass < n / S) ? S : r;
    rn.begin();
    const int down = rn.next(st_);
    mx = 0;
    if (st_ == 3) {
      for (int g = threadIdx.x; g < (N >> 3); g += blockDim.x)
        dif_group<3>(buf, g, s1, tw, nmax, down, first, last, ld, st, mx);
    } else if (st_ == 2) {
      for (int g = threadIdx.x; g < (N >> 2); g += blockDim.x)
        dif_group<2>(buf, g, s1, tw, nmax, down, first, last, ld, st, mx);
    } else if (st_ == 1) {
      for (int g = threadIdx.x; g < (N >> 1); g += blockDim.x)
        dif_group<1>(buf, g, s1, tw, nmax, down, first, last, ld, st, mx);
    } else if (threadIdx.x == 0) {
      const cx v = ld(0);
      st(0, cx{shift_down(v.x, down), shift_down(v.y, down)});
    }
    s1 -= st_;
    rn.end(mx);
  }
}

__device__ __forceinline__ int bitrev(int k, int logn) {
  return logn == 0 ? 0 : (int)(__brev((unsigned)k) >> (32 - logn));
}
__device__ __forceinline__ unsigned dexp(double v) { return ((unsigned)__double2hiint(v) >> 20) & 0x7ffu; }
__device__ __forceinline__ double fx_nan() { return __longlong_as_double(0x7ff8000000000000ll); }

enum { MODE_SYNTH = 0, MODE_ANALYSIS = 1, MODE_FUSED = 2 };
constexpr int kMaxPix = 8;
constexpr int kSMs = 152;
struct PixPtrs {
  const double* p[kMaxPix];
};

// One CTA per (map, ring pair), as in ringfft.cu; THR threads resident per SM.
template <int MODE, int NT, int THR>
__global__ void __launch_bounds__(NT, THR / NT)
k_ringfft_fx(const double2* __restrict__ F, int64_t F_stride, double* __restrict__ map_out,
             const double* __restrict__ map_in, int64_t npix, const double* __restrict__ ring_w, PixPtrs pix,
             const FftPlan* __restrict__ plans, const int* __restrict__ pair_plan,
             const int2* __restrict__ pring, const int* __restrict__ pphase,
             const int64_t* __restrict__ roff, const int4* __restrict__ tab, int64_t tw_off, int nmax, int L,
             double* __restrict__ eo, int eo_nm, int k0, int nmaps, int npair) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ unsigned s_max[3];  // exponents of the inputs (synthesis, pixels), upper word of the sums
  __shared__ unsigned s_ren[3];

  const int k = blockIdx.x;
  const int p = blockIdx.y;
  const FftPlan P = plans[pair_plan[p]];
  const int lg2 = 31 - __clz(P.n2);
  const Sbuf buf{reinterpret_cast<cx*>(smem_raw), lg2 >= 8 ? lg2 - 4 : 31};
  const int n = P.n, n2 = P.n2;
  const bool blu = P.bluestein != 0;
  const int logn = 31 - __clz(n);
  const int2 rr = pring[p];
  const bool has_s = rr.y >= 0;
  const int ph = pphase[p];
  const int64_t offN = roff[rr.x];
  const int64_t offS = has_s ? roff[rr.y] : 0;
  const int4* __restrict__ ptab = tab + P.phase;
  const int4* __restrict__ tw = tab + tw_off;
  const int4* __restrict__ chirp = tab + P.chirp;
  const int4* __restrict__ filt = tab + P.filt;
  const int tid = threadIdx.x;

  if (tid < 3) s_max[tid] = s_ren[tid] = 0;
  __syncthreads();
  Renorm rn{s_ren};
  unsigned mx = 0;
  auto bload = [&](int i) { return buf[i]; };
  // filter multiply in the last pass of a Bluestein plan's DIF transform
  auto filt_store = [&](int q, const cx& v) {
    const cx w = cmul<false>(v, filt[q]);
    mx = max(mx, hi_abs(w));
    buf[q] = w;
  };
  auto exp_scan = [&](unsigned e, int slot) {  // block maximum of exponents or upper words
    e = __reduce_max_sync(0xffffffffu, e);
    if ((tid & 31) == 0) atomicMax(&s_max[slot], e);
    __syncthreads();
    return s_max[slot];
  };

  bool bad = false;  // an input is not finite: the ring pair's results are NaN
  if (MODE == MODE_SYNTH || MODE == MODE_FUSED) {
    const double2* FN = F + k * F_stride + (int64_t)rr.x * (L + 1);
    const double2* FS = has_s ? F + k * F_stride + (int64_t)rr.y * (L + 1) : nullptr;
    unsigned e = 0;
    for (int m = tid; m <= L; m += NT) {
      const double2 a = FN[m];
      e = max(e, max(dexp(a.x), dexp(a.y)));
      if (has_s) {
        const double2 b = FS[m];
        e = max(e, max(dexp(b.x), dexp(b.y)));
      }
    }
    e = exp_scan(e, 0);
    bad = e == 0x7ffu;
    // |F| < 2^(e - 1022); a frequency sums at most na terms of each ring, and the pair's packed
    // value is below 2 sqrt(2) na of that.  Short rings with many aliases would keep too few bits of F
    // that way (47 at 4 pixels and L = 6000): they form the sums twice, first to see how large they are.
    // Differences of sums wrap, so terms that cancel may be larger than the room for their sum.
    const int na = L / n + 1 + (L + n - 1) / n, abits = 32 - __clz(na - 1);
    int kf = 61 - 2 - abits - ((int)e - 1022);
    const bool twice = abits > 4;
    auto fix = [&](double v) { return bad ? (fx_t)0 : fx_from_double(v, kf); };
    // alias sums of one frequency, as in ringfft.cu
    auto alias_sums = [&](int kk, int part, int tpk, cx& an, cx& as) {
      an = as = cx{0, 0};
      {
        int j = (kk == 0 ? 1 : 0) + part;
        for (int m = kk + j * n; m <= L; m += tpk * n, j += tpk) {
          const bool neg = ph && (j & 1);
          const double2 a = FN[m];
          const cx v{fix(a.x), -fix(a.y)};
          an = wrap_add(an, v, neg);
          if (has_s) {
            const double2 b = FS[m];
            const cx u{fix(b.x), -fix(b.y)};
            as = wrap_add(as, u, neg);
          }
        }
      }
      {
        int j = 1 + part;
        for (int m = j * n - kk; m <= L; m += tpk * n, j += tpk) {
          const bool neg = ph && (j & 1);
          const double2 a = FN[m];
          const cx v{fix(a.x), fix(a.y)};
          an = wrap_add(an, v, neg);
          if (has_s) {
            const double2 b = FS[m];
            const cx u{fix(b.x), fix(b.y)};
            as = wrap_add(as, u, neg);
          }
        }
      }
    };
    auto fold_store = [&](int kk, cx an, cx as) {
      if (ph) {
        const int4 w = ptab[kk];
        an = cmul<false>(an, w);
        as = cmul<false>(as, w);
      }
      if (kk == 0) {
        an.x += fix(FN[0].x);
        if (has_s) as.x += fix(FS[0].x);
      }
      const cx z{an.x - as.y, an.y + as.x};
      if (blu) buf[kk] = cmul<true>(cconj(z), chirp[kk]);
      else buf[bitrev(kk, logn)] = z;
    };
    // rings with fewer pixels than threads: tpk threads per frequency (ringfft.cu)
    const int scratch = n2 + n2 / 16 + 16;
    int tpk = n < NT / 2 ? NT / n : 1;
    if (scratch + 2 * NT > nmax + nmax / 16 + 16) tpk = 1;
    for (int kk = n + tid; kk < n2; kk += NT) buf[kk] = cx{0, 0};
    for (int round = twice ? 0 : 1; round < 2; ++round) {
      unsigned big = 0;
      auto take = [&](int kk, cx an, cx as) {
        if (round == 1) {
          fold_store(kk, an, as);
          return;
        }
        big = max(big, max(hi_abs(an), hi_abs(as)));
        if (kk == 0) big = max(big, max(hi_abs(fix(FN[0].x)), has_s ? hi_abs(fix(FS[0].x)) : 0u));
      };
      if (tpk == 1) {
        for (int kk = tid; kk < n; kk += NT) {
          cx an, as;
          alias_sums(kk, 0, 1, an, as);
          take(kk, an, as);
        }
      } else {
        cx* part = buf.p + scratch;
        if (tid < n * tpk) {
          cx an, as;
          alias_sums(tid % n, tid / n, tpk, an, as);
          part[2 * tid] = an;
          part[2 * tid + 1] = as;
        }
        __syncthreads();
        if (tid < n) {
          cx an{0, 0}, as{0, 0};
          for (int q = 0; q < tpk; ++q) {
            an = wrap_add(an, part[2 * (tid + q * n)], false);
            as = wrap_add(as, part[2 * (tid + q * n) + 1], false);
          }
          take(tid, an, as);
        }
      }
      if (round == 0) {
        // all components below c = 2^(64 - clz): the packed value's modulus is below 7 c (a frequency
        // and its m = 0 term of both rings, turned by their phases)
        const unsigned h = exp_scan(big, 2);
        kf += max(0, min(abits, __clz(h) - 6));
      }
    }
    __syncthreads();
    const double* pk = MODE == MODE_FUSED ? pix.p[k] : nullptr;
    double* mo = MODE == MODE_SYNTH ? map_out + k * npix : nullptr;
    unsigned pe = 0;  // largest exponent of the multiplied pixels
    auto pixel_store = [&](int t, cx z) {
      if (blu) {
        if (t >= n) return;
        z = cconj(cmul<true>(z, chirp[t]));
      }
      const int ex = rn.shifted + (blu ? P.fexp : 0) - kf;  // every pass's shift is counted by now
      double zx = bad ? fx_nan() : fx_value(z.x, ex), zy = bad ? fx_nan() : fx_value(z.y, ex);
      if (MODE == MODE_SYNTH) {
        mo[offN + t] = zx;
        if (has_s) mo[offS + t] = zy;
        return;
      }
      zx = zx * pk[offN + t];
      zy = has_s ? zy * pk[offS + t] : 0.0;
      pe = max(pe, max(dexp(zx), dexp(zy)));
      *reinterpret_cast<double2*>(&buf[t]) = make_double2(zx, zy);
    };
    if (!blu) {
      fft_dit<true>(buf, n, tw, nmax, rn, mx, bload, pixel_store);
    } else {
      fft_dif(buf, n2, tw, nmax, rn, mx, bload, filt_store);
      fft_dit<true>(buf, n2, tw, nmax, rn, mx, bload, pixel_store);
    }
    if (MODE == MODE_SYNTH) return;
    pe = __reduce_max_sync(0xffffffffu, pe);
    if ((tid & 31) == 0) atomicMax(&s_max[1], pe);
    __syncthreads();
  }
  const double* mi = MODE == MODE_ANALYSIS ? map_in + k * npix : nullptr;
  if (MODE == MODE_ANALYSIS) {
    unsigned e = 0;
    for (int t = tid; t < n; t += NT) {
      e = max(e, dexp(mi[offN + t]));
      if (has_s) e = max(e, dexp(mi[offS + t]));
    }
    exp_scan(e, 1);
  }
  // forward DFT; its first pass reads the pixels (analysis: maps, fused: the buffer)
  const unsigned e1 = s_max[1];
  bad |= e1 == 0x7ffu;
  const int kp = 60 - ((int)e1 - 1022);
  auto pixel_load = [&](int t) {
    if (t >= n || bad) return cx{0, 0};
    double2 v;
    if (MODE == MODE_ANALYSIS) v = make_double2(mi[offN + t], has_s ? mi[offS + t] : 0.0);
    else v = *reinterpret_cast<const double2*>(&buf[t]);
    const cx z{fx_from_double(v.x, kp), fx_from_double(v.y, kp)};
    return blu ? cmul<true>(z, chirp[t]) : z;
  };
  auto bstore = [&](int i, const cx& v) { buf[i] = v; };
  rn.gain = rn.shifted = 0;
  if (!blu) {
    fft_dif(buf, n, tw, nmax, rn, mx, pixel_load, bstore);
  } else {
    fft_dif(buf, n2, tw, nmax, rn, mx, pixel_load, filt_store);
    auto chirp_store = [&](int t, const cx& c) {
      if (t < n) buf[t] = cmul<true>(c, chirp[t]);
    };
    fft_dit<true>(buf, n2, tw, nmax, rn, mx, bload, chirp_store);
  }
  const int ex = rn.shifted + (blu ? P.fexp : 0) - kp;  // values = fixed-point numbers times 2^ex

  // unfold (ringfft.cu), without the sqrt(2) of m > 0: G_m = exp(-i m phi0) X_{m mod n}, results
  // (Re G, -Im G) of each ring, written as north + south and north - south
  const double wN = (MODE == MODE_ANALYSIS && ring_w) ? ring_w[rr.x] : 1.0;  // the pair's rings agree
  const int kg = k0 + k, ch = kg / eo_nm, j = kg - ch * eo_nm;
  const int nmc = min(eo_nm, nmaps - ch * eo_nm), PP = 2 * nmc;
  double* ec = eo + (int64_t)ch * eo_nm * (L + 1) * npair * 4 + (int64_t)p * 2 * PP + 2 * j;
  for (int m = tid; m <= L; m += NT) {
    const int kk = m % n;
    const int kc = (kk == 0) ? 0 : n - kk;
    const cx zk = buf[blu ? kk : bitrev(kk, logn)];
    const cx zc = cconj(buf[blu ? kc : bitrev(kc, logn)]);
    const cx a = zk + zc, b = zk - zc;
    cx gn{(a.x + 1) >> 1, (a.y + 1) >> 1};
    cx gs{(b.y + 1) >> 1, -((b.x + 1) >> 1)};
    if (ph) {
      const int4 w = ptab[kk];
      gn = cmul<true>(gn, w);
      gs = cmul<true>(gs, w);
      if ((m / n) & 1) {
        gn = cx{-gn.x, -gn.y};
        gs = cx{-gs.x, -gs.y};
      }
    }
    cx on{gn.x, m == 0 ? 0 : -gn.y}, os{gs.x, m == 0 ? 0 : -gs.y};
    if (!has_s) os = cx{0, 0};
    const cx ev = on + os, od = on - os;
    double2 vev = make_double2(fx_value(ev.x, ex), fx_value(ev.y, ex));
    double2 vod = make_double2(fx_value(od.x, ex), fx_value(od.y, ex));
    if (MODE == MODE_ANALYSIS && ring_w) {
      vev.x *= wN;
      vev.y *= wN;
      vod.x *= wN;
      vod.y *= wN;
    }
    if (bad) vev = vod = make_double2(fx_nan(), fx_nan());
    double* e = ec + (int64_t)m * npair * 2 * PP;
    *reinterpret_cast<double2*>(e) = vev;
    *reinterpret_cast<double2*>(e + PP) = vod;
  }
}

template <int MODE, int NT, int THR>
int launch_thr(const Grid& g, int nmaps, const void* F, double* map_out, const double* map_in, int weighted,
              const void* const* pix, void* eo, cudaStream_t s) {
  const size_t sm = (size_t)(g.nmax2 + g.nmax2 / 16 + 16) * sizeof(cx);
  if (sm > 227 * 1024) {
    set_error("ring FFT needs %zu bytes of shared memory (ring length %d) at this precision", sm, g.max_n);
    return CMBWS_ERR_ARG;
  }
  auto kern = k_ringfft_fx<MODE, NT, THR>;
  CMBWS_TRY(ensure_dyn_smem((const void*)kern, sm));
  const int64_t fs = (int64_t)g.nring * (g.lmax + 1);
  const double* rw = (MODE == MODE_ANALYSIS && weighted) ? g.ring_w64.as<double>() : nullptr;
  for (int k0 = 0; k0 < nmaps; k0 += kMaxPix) {
    const int nm = nmaps - k0 < kMaxPix ? nmaps - k0 : kMaxPix;
    PixPtrs pp{};
    if (MODE == MODE_FUSED)
      for (int i = 0; i < nm; ++i) pp.p[i] = (const double*)pix[k0 + i];
    dim3 grd(nm, g.npair);
    const double fb = (double)g.nring * (g.lmax + 1) * 16, pb = (double)g.npix * 8;
    ProfScope ps(PROF_FFT, s, 1, byte_work(nm * ((MODE == MODE_FUSED ? 2.0 : 1.0) * fb + pb)));
    kern<<<grd, NT, sm, s>>>(F ? (const double2*)F + k0 * fs : nullptr, fs,
                             map_out ? map_out + k0 * g.npix : nullptr,
                             map_in ? map_in + k0 * g.npix : nullptr, g.npix, rw, pp,
                             g.plans_d.as<FftPlan>(), g.pair_plan.as<int>(), g.pair_ring.as<int2>(),
                             g.pair_phase.as<int>(), g.ring_off.as<int64_t>(), g.fftfx.as<int4>(), g.tw_off,
                             g.nmax2, g.lmax, (double*)eo, eo_maps(CMBWS_FP64), k0, nmaps, g.npair);
    CMBWS_LAUNCH_CHECK();
  }
  return CMBWS_OK;
}

// Registers: 128 per thread keep the transforms free of spills, at 512 threads per SM; 85, at 768, hide
// more latency but spill.  The second form is taken where its larger waves are fewer: 5 maps on a GL
// grid of 512 rings (1280 CTAs of 128 threads, 3 waves -> 2) 337 -> 270 us, 3 maps (768, 2 -> 1)
// 240 -> 177 us for both directions, Nside 512 (3072 of 256, 11 -> 7) 842 -> 734 us; on grids of one
// wave it is slower (solve with 96 CTAs per transform: 959 -> 1032 us).
template <int MODE, int NT>
int launch_nt(const Grid& g, int nmaps, const void* F, double* map_out, const double* map_in, int weighted,
              const void* const* pix, void* eo, cudaStream_t s) {
  constexpr int64_t lo = kSMs * (512 / NT), hi = kSMs * (768 / NT);  // CTAs of a wave
  const int64_t n = (int64_t)g.npair * (nmaps < kMaxPix ? nmaps : kMaxPix);
  if constexpr (hi > lo)
    if ((n + hi - 1) / hi < (n + lo - 1) / lo)
      return launch_thr<MODE, NT, 768>(g, nmaps, F, map_out, map_in, weighted, pix, eo, s);
  return launch_thr<MODE, NT, 512>(g, nmaps, F, map_out, map_in, weighted, pix, eo, s);
}

// threads per CTA by the transform buffer, as in ringfft.cu
template <int MODE>
int launch(const Grid& g, int nmaps, const void* F, double* map_out, const double* map_in, int weighted,
           const void* const* pix, void* eo, cudaStream_t s) {
  if (g.nmax2 >= 8192) return launch_nt<MODE, 512>(g, nmaps, F, map_out, map_in, weighted, pix, eo, s);
  if (g.nmax2 >= 4096) return launch_nt<MODE, 256>(g, nmaps, F, map_out, map_in, weighted, pix, eo, s);
  return launch_nt<MODE, 128>(g, nmaps, F, map_out, map_in, weighted, pix, eo, s);
}

}  // namespace

int ringfft_fx_synth(const Grid& g, int nmaps, const void* F, double* map, cudaStream_t s) {
  return launch<MODE_SYNTH>(g, nmaps, F, map, nullptr, 0, nullptr, nullptr, s);
}
int ringfft_fx_analysis(const Grid& g, int nmaps, const double* map, int weighted, void* eo, cudaStream_t s) {
  return launch<MODE_ANALYSIS>(g, nmaps, nullptr, nullptr, map, weighted, nullptr, eo, s);
}
int ringfft_fx_fused(const Grid& g, int nmaps, const void* F, const void* const* pix, void* eo,
                     cudaStream_t s) {
  return launch<MODE_FUSED>(g, nmaps, F, nullptr, nullptr, 0, pix, eo, s);
}

}  // namespace cmbws
