// FP64 Legendre stage (CMBWS_FP64): the recurrence in 64-bit fixed
// point on the CUDA cores, the contraction on the tcgen05 tensor cores over 8-bit digits with
// exact sums.  The arithmetic, its digits and their error are described in fixed.h.
//
// Both stages are products with Lambda[pair][l] = mu_l(theta_pair) (Sec. 2.1):
//   synthesis   D[pair][col] = sum_l Lambda[pair][l] B[l][col], col = parity(l - m) W + part;
//   adjoint     D[l][col] = sum_pairs Lambda[pair][l] B[pair][col], col = h W + part, h = 0 the
//               even part (north + south) and h = 1 the odd one; row l reads its own parity.  The
//               real parts of all maps come first: a warp takes either them or the imaginary ones
//               (half the columns to read, no spills: one map at L = 1000 917 -> 836 us with the FFT).
// W is 8 (up to 4 maps) or 16 (up to 8 maps): the recurrence, which is most of the work, serves all
// of them.  The 8 digits of Lambda are the A operand (shared memory, one tile per digit), those of
// the coefficients or ring parts the B operand (8 x 2 W rows); digit i of A times the digits
// 0..7 - i of B accumulate into columns 2 W i.. of the accumulator, so that block s of 2 W columns
// holds the sum over i + j = s.  Every 64 terms the blocks are read from tensor memory and added
// as integers.
#include <atomic>
#include <climits>
#include <type_traits>

#include "common.h"
#include "fixed.h"
#include "tcgen05.h"

namespace cmbws {

namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kM = 128;              // MMA rows: ring pairs (synthesis) or values of l (adjoint)
constexpr int kNT = 2 * kM;          // threads per CTA: two per row
constexpr int kMaxDevices = 64;

// Column layout for up to NM maps.  Up to 4 maps have an instance each; 5 and 6 maps share one, 7 and 8
// another.  Eight columns per parity up to 4 maps keep three CTAs on an SM, which the recurrence's
// latency needs; 16 columns for 5 to 8 maps give up one of them for half the recurrences.  Against
// launches of 4 maps: analysis of 5 maps at L = 131 88 -> 60 us, an apply of A on 5 GL grids at
// L = 511 969 -> 810 us, one on grids of 9 maps at L = 297 1114 -> 902 us.
template <int NM>
struct Cols {
  static constexpr int W = NM <= 4 ? 8 : 16;           // columns per parity
  static constexpr int kDig = 2 * W * 32;              // bytes of one digit of B: 2 W rows x 16 halves
  static constexpr int kBStep = kFxDig * kDig;         // one K step of B
  static constexpr uint32_t kTmem = kFxBlk * 2 * W;    // accumulator columns
  static constexpr int kCtas = NM <= 4 ? 3 : 2;        // CTAs per SM (256 columns: two)
};

__device__ unsigned int g_fx_status = 0;  // bit 0: a bounded mbarrier wait ran out
// Test support (cmbws_testing_stall_waits), by device: when > 0, every CTA first waits at most this many
// SM clocks on an mbarrier phase that nothing completes, so the wait runs out.  A kernel argument: reading
// it from device memory would be on the way of every short launch.
std::atomic<long long> g_stall[kMaxDevices];
long long stall_of(const Grid& g) {
  return g.device < kMaxDevices ? g_stall[g.device].load(std::memory_order_relaxed) : 0;
}

// kind::f16, FP16 A and B, FP32 D, M = 128, N = ncol; A K-major or MN-major, B K-major
__device__ __forceinline__ void mma_f16(uint32_t d, uint64_t adesc, uint64_t bdesc, int ncol, bool mn,
                                        uint32_t acc) {
  const uint32_t idesc = (1u << 4) | (mn ? 1u << 15 : 0u) | ((uint32_t)(ncol >> 3) << 17) | (8u << 24);
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(d),
      "l"(adesc), "l"(bdesc), "r"(idesc), "r"(acc)
      : "memory");
}
// One K step: digit i of A (tiles atile bytes apart) times the digits 0..7 - i of B into blocks
// i..7; `first` clears the accumulator (digit 0 writes all blocks).
template <typename C>
__device__ __forceinline__ void mma_step(uint32_t d, uint32_t ab, int atile, uint32_t alb, uint32_t asb,
                                         uint32_t bb, bool mn, bool first) {
  constexpr int N = 2 * C::W;
  const uint64_t b0 = smem_desc(bb, 128, 256);
  mma_f16(d, smem_desc(ab, alb, asb), b0, N * kFxBlk, mn, first ? 0u : 1u);
#pragma unroll
  for (int i = 1; i < kFxDig; ++i)
    mma_f16(d + N * i, smem_desc(ab + i * atile, alb, asb), b0, N * (kFxBlk - i), mn, 1u);
}

template <uint32_t COLS>
__device__ __forceinline__ void tmem_alloc(uint32_t* slot) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_addr(slot)),
               "n"(COLS)
               : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
}
template <uint32_t COLS>
__device__ __forceinline__ void tmem_free(uint32_t tb) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tb), "n"(COLS) : "memory");
}
template <int W>
__device__ __forceinline__ void tmem_ld(uint32_t taddr, uint32_t (&d)[W]) {
  if constexpr (W == 4) tmem_ld4(taddr, d);
  else if constexpr (W == 8) tmem_ld8(taddr, d);
  else tmem_ld16(taddr, d);
}

// digit words of zero (byte 7 is stored plus 128)
__device__ __forceinline__ unsigned zero_digit(int i) { return i == 0 ? 0x00800080u : 0u; }

// Eight values of l of one pair as digits: per digit one 16-byte row of A (8 halves), tiles `tile`
// bytes apart.  co: the recurrence coefficients; la: the first l; ls: where the pair starts (s0 the
// values there); skip: the state already holds the first two values; wait(): the previous stage's
// MMAs have read the tile.
template <int Q>
using Half = std::integral_constant<int, Q>;
template <typename W>
__device__ __forceinline__ void fx_walk8(FxState& s, const int4* co, unsigned xh, unsigned xl, int la,
                                         int ls, const FxState& s0, bool skip, unsigned char* row,
                                         int tile, W&& wait) {
  // warp-uniform: a pair starts here, or still carries an exponent
  if (__any_sync(kFull, s.e > 0 || (ls >= la && ls < la + 8))) {
    wait();
#pragma unroll 1
    for (int j = 0; j < 8; j += 2) {
      if (!skip || j > 0) fx_step2_slow(s, co[j], co[j + 1], xh, xl, ls == la + j, s0);
      const fxu_t a = fx_bytes(fx_emit(s.V2, s.e)), b = fx_bytes(fx_emit(s.V1, s.e));
      auto put = [&](auto q) {
        unsigned d0, d1;
        fx_digits2<q.value>(a, b, d0, d1);
        *reinterpret_cast<unsigned*>(row + (6 - 2 * q.value) * tile + 2 * j) = d0;
        *reinterpret_cast<unsigned*>(row + (7 - 2 * q.value) * tile + 2 * j) = d1;
      };
      put(Half<0>{}), put(Half<1>{}), put(Half<2>{}), put(Half<3>{});
    }
    return;
  }
  fxu_t v[8];
#pragma unroll
  for (int j = 0; j < 8; j += 2) {
    if (j > 0 || !skip) s.step2(co[j], co[j + 1], xh, xl);
    v[j] = fx_bytes(s.V2);
    v[j + 1] = fx_bytes(s.V1);
  }
  wait();
  // two digits of all eight values at a time: the values take half the registers of their digits
  auto put = [&](auto q) {
    uint4 r0, r1;
    fx_digits2<q.value>(v[0], v[1], r0.x, r1.x);
    fx_digits2<q.value>(v[2], v[3], r0.y, r1.y);
    fx_digits2<q.value>(v[4], v[5], r0.z, r1.z);
    fx_digits2<q.value>(v[6], v[7], r0.w, r1.w);
    *reinterpret_cast<uint4*>(row + (6 - 2 * q.value) * tile) = r0;
    *reinterpret_cast<uint4*>(row + (7 - 2 * q.value) * tile) = r1;
  };
  put(Half<0>{}), put(Half<1>{}), put(Half<2>{}), put(Half<3>{});
}

__device__ __forceinline__ int digit_sum(uint32_t d) {
  return __float2int_rn(__uint_as_float(d) * 16777216.f);  // FP16 subnormals: units of 2^-24
}

__device__ __forceinline__ double fx_nan() { return __longlong_as_double(0x7ff8000000000000ll); }

// ---- synthesis ----
constexpr int kSynK = 16;                        // values of l per stage (one K step)
constexpr int kSynPeriod = 8;                    // stages between two reads: 64 terms per parity
constexpr int kSynTile = kM * kSynK * 2;         // one digit of A
constexpr int kSynA = kFxDig * kSynTile;
template <typename C>
struct SynLayout {
  static constexpr int kA = 0;                      // also the odd sums at the end: double[2 NM][128]
  static constexpr int kB = kSynA;                  // two stages of B
  static constexpr int kCoef = kB + 2 * C::kBStep;  // int4[2][16]
  static constexpr int kCorr = kCoef + 2 * kSynK * 16;  // fxu_t[2 W][2]
  static constexpr int kBar = kCorr + 2 * C::W * 16;    // uint64_t[2]
  static constexpr int kMisc = kBar + 16;           // tensor memory base, bad flag
  static constexpr int kExp = kMisc + 16;           // exponents [3][8]
  static constexpr int kScale = kExp + 96;          // scales of the pairs (uint8)
  static constexpr int kBytes = kScale + kM;
};

// Steep spectra.  One scale per (m, map) holds a coefficient to 2^-61 of the largest one that the rings of
// the CTA can see, where FP64 arithmetic holds it to 2^-53 of itself.  That is enough for a ring's map if
// the largest one is below 2^8 of what lights the ring anyway: its coefficients of m = 0, whose Legendre
// values are of order one at every l and ring (the first 128 and 128 from the whole range stand for them),
// or those of this m from where the ring's values are of order one (l sin(theta) = m; for the CTA's ring
// nearest the pole).  Only spectra without much at m = 0 that fall by more than 2^8 along this m fail
// both; their sums are taken in FP64 arithmetic instead (from the start at 1e-30), by two threads per ring
// pair, one for each parity.
constexpr int kSteep = 8;
// Sum over l of mu_l a_l with l - m of parity par; a, A at index l; ls, st: the pair's start.
__device__ __noinline__ double2 synth_fp64(const double2* a, const double* A, double y, int ls, double2 st,
                                           int L, int par) {
  double re = 0.0, im = 0.0, m2 = st.x, m1 = st.y;
  for (int l = ls; l <= L; l += 2) {
    if (l + par <= L) {
      const double mu = par ? m1 : m2;
      const double2 v = a[l + par];
      re = fma(mu, v.x, re);
      im = fma(mu, v.y, im);
    }
    if (l + 2 > L) break;
    m2 = fma(-A[l + 2], y, A[l + 2]) * m1 - m2;
    m1 = l + 3 <= L ? fma(-A[l + 3], y, A[l + 3]) * m2 - m1 : 0.0;
  }
  return make_double2(re, im);
}

// Two threads per ring pair (row of A) walk l upwards: one from the first start of the CTA's pairs,
// one from the checkpoint in the middle of the rest (half the chain, twice the warps to hide the
// recurrence's latency).  Per stage each writes the digits of 8 values of l as one 16-byte row per
// digit tile (consecutive threads are 16 bytes apart); every second stage it converts one
// coefficient part to digits of B.  One thread issues the stage's MMAs after its barrier; they read
// the tile while the threads compute the next values in registers.
// Bound by the dispatch of integer instructions (50 per element, about half of them at half rate; tensor
// pipe 15 %).  Against the recurrence and sums on the FP64 pipe, Nside 1024, L = 3071, 3 maps: 94.6 ->
// 19.9 ms (19.1 with 7 digits and one scale per m, which lost precision: fixed.h).  An early form with one
// chain per row and 128 threads took 19.0 ms there where two chains took 19.9 (not tried since), but
// grids of few ring pairs wait for that chain.
template <int NM>
__global__ void __launch_bounds__(kNT, Cols<NM>::kCtas)
k_leg_synth_fx(const double2* __restrict__ alm, int64_t alm_stride, const double* __restrict__ Acoef,
               const uint8_t* __restrict__ sx, const int* __restrict__ ls_tab,
               const int* __restrict__ tmin, const ulonglong2* __restrict__ st, const uint64_t* __restrict__ xfx,
               const ulonglong2* __restrict__ ck, const int64_t* __restrict__ ck_base,
               const int2* __restrict__ pring, const int* __restrict__ ls64, const double2* __restrict__ st64,
               const double* __restrict__ y64, double2* __restrict__ F, int64_t F_stride, int L, int npair,
               int R, int nmaps, long long stall) {
  using C = Cols<NM>;
  using LY = SynLayout<C>;
  constexpr int P = 2 * NM, W = C::W;
  const int nm = NM <= 4 ? NM : nmaps;
  extern __shared__ __align__(1024) unsigned char sm[];
  int4* s_coef = reinterpret_cast<int4*>(sm + LY::kCoef);
  fxu_t* s_corr = reinterpret_cast<fxu_t*>(sm + LY::kCorr);
  uint64_t* mbar = reinterpret_cast<uint64_t*>(sm + LY::kBar);
  uint32_t* s_tb = reinterpret_cast<uint32_t*>(sm + LY::kMisc);
  int* s_bad = reinterpret_cast<int*>(sm + LY::kMisc + 4);
  // exponents per map: largest coefficient from the group's first start on, from s_ehi's l on, of m = 0
  unsigned* s_emax = reinterpret_cast<unsigned*>(sm + LY::kExp);
  unsigned *s_ehi = s_emax + 8, *s_e0 = s_emax + 16;

  const int tid = threadIdx.x, warp = tid >> 5;
  const int row = tid & (kM - 1), chain = tid >> 7;  // chain: warp-uniform
  const int m = blockIdx.y;
  const int64_t lmo = lm_off(L, m) - m;  // index of (m, l) is lmo + l

  if (tid < 24) s_emax[tid] = 0;
  if (tid == 0) {
    *s_bad = 0;
    mbar_init(&mbar[0], 1);
    mbar_init(&mbar[1], 1);
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  }
  // of a group: the first start, and the l from where the Legendre values of the ring nearest the pole are
  // of order one (loaded ahead of their use)
  int lo_r, hi_r;
  auto group_range = [&](int r) {
    const int p0 = (blockIdx.x * R + r) * kM;
    const int ntm = (npair + kTileMinPT - 1) / kTileMinPT, t0 = p0 / kTileMinPT;
    const float y0 = p0 < npair ? (float)y64[p0] : 1.f;
    lo_r = L + 1;
    for (int t = t0; t < min(ntm, t0 + kM / kTileMinPT); ++t) lo_r = min(lo_r, tmin[(int64_t)m * ntm + t]);
    hi_r = (int)fminf((float)L, ceilf((float)m * rsqrtf(fmaxf(y0 * (2.f - y0), 1e-30f))));
  };
  group_range(0);
  auto exp2 = [](double2 v) {
    return max((unsigned)__double2hiint(v.x) & 0x7fffffffu, (unsigned)__double2hiint(v.y) & 0x7fffffffu) >> 20;
  };
  // zero B (columns of the other parity and of absent maps stay zero)
  for (int i = tid; i < 2 * C::kBStep / 16; i += kNT)
    reinterpret_cast<uint4*>(sm + LY::kB)[i] = make_uint4(0, 0, 0, 0);
  if (stall > 0 && tid == 0 && !mbar_wait(&mbar[1], 0, stall)) *s_bad = 1;
  __syncwarp();
  if (warp == 0) tmem_alloc<C::kTmem>(s_tb);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tb = *s_tb;
  const uint32_t lane_base = (uint32_t)((warp & 3) * 32) << 16;

  // this thread's coefficient part of a stage (W = 8: of the stages t with t mod 2 = chain): value k
  // of l (0..7 of the first chain, 8..15 of the second), part q (re / im of each map)
  constexpr int kBEvery = W == 8 ? 2 : 1;
  const int bk = tid & 15, bq = (tid >> 4) & (W - 1);
  const bool bon = bq < 2 * nm;
  const double* bsrc = reinterpret_cast<const double*>(alm + (bq >> 1) * alm_stride + lmo) + (bq & 1);
  unsigned char* bdst = sm + LY::kB + (bk & 1) * W * 32 + (bk >> 3) * 128 + (bq >> 3) * 256 + (bq & 7) * 16 +
                        (bk & 7) * 2;
  unsigned char* arow = sm + LY::kA + chain * (kSynTile / 2) + row * 16;

  int gs = 0;  // stages issued by this CTA
  bool bad = false;
  for (int r = 0; r < R; ++r) {
    const int p = (blockIdx.x * R + r) * kM + row;
    const bool valid = p < npair;
    const int ls = valid ? ls_tab[(int64_t)m * npair + p] : INT_MAX;
    const uint64_t x = valid ? xfx[p] : 0;
    const unsigned xh = (unsigned)(x >> 32), xl = (unsigned)x;
    if (!chain) sm[LY::kScale + row] = valid ? sx[(int64_t)m * npair + p] : 0;
    FxState s0;  // the pair's start values
    if (ls <= L) {
      s0 = fx_unpack(st[(int64_t)m * npair + p]);
      if ((ls - m) & 2) fx_negate(s0);
    }
    if (tid < 4 * W) s_corr[tid] = 0;
    const int wlo = __reduce_min_sync(kFull, ls);
    if (r > 0) group_range(r);
    const int lo = lo_r, hi = hi_r;
    // scale of each map: the largest exponent among this m's coefficients from lo on (any that is not
    // finite counts)
    if (r > 0) {
      if (tid < 16) s_emax[tid] = 0;
      __syncthreads();
    }
#pragma unroll
    for (int k = 0; k < NM; ++k) {
      if (k >= nm) break;
      unsigned e = 0, eh = 0, e0 = 0;
      if (r == 0) {
        const int l = chain ? row * ((L + kM) / kM) : row;
        if (l <= L) e0 = exp2(alm[k * alm_stride + l]);
      }
#pragma unroll 4
      for (int l = m + tid; l <= L; l += kNT) {
        const unsigned x = exp2(alm[k * alm_stride + lmo + l]);
        if (l >= lo || x == 0x7ffu) e = max(e, x);
        if (l >= hi) eh = max(eh, x);
      }
      e = __reduce_max_sync(kFull, e);
      eh = __reduce_max_sync(kFull, eh);
      e0 = __reduce_max_sync(kFull, e0);
      if ((tid & 31) == 0) {
        atomicMax(&s_emax[k], e);
        atomicMax(&s_ehi[k], eh);
        atomicMax(&s_e0[k], e0);
      }
    }
    __syncthreads();
    auto steep = [&](int k) {
      return s_emax[k] < 0x7ffu && s_emax[k] > max(s_ehi[k], s_e0[k]) + kSteep;
    };
    bool all_steep = true;
    for (int k = 0; k < nm; ++k) all_steep &= steep(k);
    const int eb = bon ? (int)s_emax[bq >> 1] - 1022 : 0;  // |a| < 2^eb; 1025 if not finite
    // rows of pairs that have not started: zero digits
#pragma unroll
    for (int i = 0; i < kFxDig; ++i) {
      const unsigned z = zero_digit(i);
      *reinterpret_cast<uint4*>(arow + i * kSynTile) = make_uint4(z, z, z, z);
    }
    // the second chain starts at a checkpoint l = lm near the middle of lo..L (past L: none)
    const int cm = ((lo + L) / 2 - m + kFxChunk / 2) / kFxChunk;
    int lm = m + kFxChunk * cm;
    if (lm <= lo) lm += kFxChunk;
    const int len = lo <= L && !all_steep ? max(min(lm, L + 1) - lo, L + 1 - lm) : 0;
    const int nst = (len + kSynK / 2 - 1) / (kSynK / 2);
    // l of value k (0..15) of stage t, or -1
    auto l_of = [&](int t, int k) {
      const int l = (k < 8 ? lo : lm - 8) + 8 * t + k;
      return t < nst && l <= L && (k >= 8 || l < lm) ? l : -1;
    };
    auto load_a = [&](int t) {  // coefficient part of stage t
      const int l = l_of(t, bk);
      return (bon && eb < 1025 && l >= 0) ? bsrc[2 * l] : 0.0;
    };
    auto load_c = [&](int t) {  // recurrence coefficient of stage t (16 threads)
      const int l = l_of(t, tid & 15);
      return l >= 0 ? Acoef[lmo + l] : 0.0;
    };
    const bool con = tid >= 112 && tid < 128;
    const bool neg = (((bk < 8 ? lo - m : 0) + bk) & 2) != 0;  // sigma of this thread's values of l
    double anext = load_a(kBEvery == 2 ? chain : 0), cnext = con ? load_c(0) : 0.0;
    if (con) s_coef[tid & 15] = fx_coef(cnext);
    cnext = con ? load_c(1) : 0.0;
    __syncthreads();

    FxState s;
    if (chain && valid && lm <= L) {
      s = fx_unpack(ck[ck_base[m] + (int64_t)p * ((L - m + kFxChunk) / kFxChunk) + (lm - m) / kFxChunk]);
    }
    const int la0 = chain ? lm : lo;                   // first l of this thread's chain
    const int lst = chain && ls <= lm ? INT_MAX : ls;  // where the pair starts in it
    FxSum acc[P];  // sums of the parity `chain`
    fx_t shi = 0, slo = 0;
    for (int t = 0; t < nst; ++t, ++gs) {
      if (con) {  // coefficients of the next stage
        s_coef[((t + 1) & 1) * kSynK + (tid & 15)] = fx_coef(cnext);
        cnext = load_c(t + 2);
      }
      if (kBEvery == 1 || (t & 1) == chain) {
        const double av = anext;
        anext = load_a(t + kBEvery);
        if (bon) {  // B of this stage: its buffer was read two stages ago
          const fx_t v = fx_from_double(neg ? -av : av, kFxABits - eb);
          unsigned dig[kFxDig];
          fx_coef_digits(v, 0, dig);
          shi += v >> 30;
          slo += v & ((1 << 30) - 1);
#pragma unroll
          for (int j = 0; j < kFxDig; ++j)
            *reinterpret_cast<unsigned short*>(bdst + (gs & 1) * C::kBStep + j * C::kDig) = (unsigned short)dig[j];
        }
      }
      auto wait = [&]() {  // the previous stage's MMAs have read the tile
        if (gs >= 1 && !*s_bad && !mbar_wait(&mbar[0], (gs - 1) & 1)) bad = true;
      };
      if (wlo < la0 + 8 * t + 8)  // some pair of the warp has started
        fx_walk8(s, s_coef + (t & 1) * kSynK + 8 * chain, xh, xl, la0 + 8 * t, lst, s0, chain && t == 0,
                 arow, kSynTile, wait);
      else
        wait();
      fence_smem_async();
      tc_fence_before();
      if (bad) atomicOr(s_bad, 1);
      __syncthreads();
      const bool first = t % kSynPeriod == 0;
      if (tid == 0 && !*s_bad) {
        tc_fence_after();
        mma_step<C>(tb, smem_addr(sm + LY::kA), kSynTile, kSynTile / 2, 128,
                 smem_addr(sm + LY::kB + (gs & 1) * C::kBStep), false, first);
        tc_commit(&mbar[0]);
      }
      if (t % kSynPeriod == kSynPeriod - 1 || t == nst - 1) {
        if (!*s_bad && !mbar_wait(&mbar[0], gs & 1)) bad = true;
        tc_fence_after();
        int prev[P];
#pragma unroll
        for (int b = 0; b < kFxBlk; ++b) {
          uint32_t d[W];
          tmem_ld<W>(tb + lane_base + 2 * W * b + W * chain, d);
          tmem_ld_wait();
#pragma unroll
          for (int q = 0; q < P; ++q) acc[q].add(b, digit_sum(d[q]), prev[q]);
        }
        tc_fence_before();  // read before the next stage's MMAs, which follow its barrier
      }
    }
    if (bon) {
      atomicAdd(&s_corr[2 * ((bk & 1) * W + bq)], (fxu_t)shi);
      atomicAdd(&s_corr[2 * ((bk & 1) * W + bq) + 1], (fxu_t)slo);
    }
    if (bad) atomicOr(s_bad, 1);
    __syncthreads();
    const bool failed = *s_bad != 0;
    const int S = sm[LY::kScale + row];
    double v[P];
    double* s_odd = reinterpret_cast<double*>(sm + LY::kA);  // [part][row]; all MMAs are done
#pragma unroll
    for (int q = 0; q < P; ++q)
      v[q] = acc[q].value((fx_t)s_corr[2 * (W * chain + q)], (fx_t)s_corr[2 * (W * chain + q) + 1],
                          (int)s_emax[q >> 1] - 1022 - S - 6);
#pragma unroll
    for (int k = 0; k < NM; ++k) {
      if (k >= nm || !steep(k)) continue;
      double2 f = make_double2(0.0, 0.0);
      const int l1 = valid ? ls64[(int64_t)m * npair + p] : INT_MAX;
      if (l1 <= L)
        f = synth_fp64(alm + k * alm_stride + lmo, Acoef + lmo, y64[p], l1, st64[(int64_t)m * npair + p], L, chain);
      v[2 * k] = f.x;
      v[2 * k + 1] = f.y;
    }
#pragma unroll
    for (int q = 0; q < P; ++q) {
      // a map with a non-finite coefficient, and a timed-out wait, give NaN
      if (m > 0) v[q] *= 0.70710678118654752440;  // the ring FFT's 1 / sqrt(2)
      if ((s_emax[q >> 1] == 0x7ffu && ls <= L) || failed) v[q] = fx_nan();
      if (chain) s_odd[q * kM + row] = v[q];
    }
    __syncthreads();
    if (valid && !chain) {
      const int2 rr = pring[p];
#pragma unroll
      for (int k = 0; k < NM; ++k) {
        if (k >= nm) break;
        const double ox = s_odd[2 * k * kM + row], oy = s_odd[(2 * k + 1) * kM + row];
        F[k * F_stride + (int64_t)rr.x * (L + 1) + m] = make_double2(v[2 * k] + ox, v[2 * k + 1] + oy);
        if (rr.y >= 0)
          F[k * F_stride + (int64_t)rr.y * (L + 1) + m] = make_double2(v[2 * k] - ox, v[2 * k + 1] - oy);
      }
    }
    __syncthreads();  // s_corr and the A rows are reset for the next group
  }
  if (tid == 0 && *s_bad) atomicOr(&g_fx_status, 1u);
  if (warp == 0) tmem_free<C::kTmem>(tb);
}

// Tiles: groups of 128 ring pairs per CTA, taken one after the other (the autotuner's list of the
// synthesis; without it one group per CTA, variant 1).
constexpr int kFxTiles = 4;
template <int NM>
int launch_synth_variant(int v, int nm, const Grid& g, const void* alm, int64_t as, void* F, int64_t fs,
                         cudaStream_t s) {
  using LY = SynLayout<Cols<NM>>;
  constexpr int kR[kFxTiles] = {2, 1, 8, 4};
  const int R = kR[v];
  const int L = g.lmax;
  dim3 grd((g.npair + kM * R - 1) / (kM * R), L + 1);
  auto kern = k_leg_synth_fx<NM>;
  CMBWS_TRY(ensure_dyn_smem((const void*)kern, LY::kBytes));
  ProfScope ps(PROF_LEG_SYNTH, s, 1, leg_work(g, nm));
  kern<<<grd, kNT, LY::kBytes, s>>>((const double2*)alm, as, g.A64.as<double>(), g.sx.as<uint8_t>(),
                                    g.lsx.as<int>(), g.lsx_tmin.as<int>(), g.stx.as<ulonglong2>(),
                                    g.xfx.as<uint64_t>(), g.ckx.as<ulonglong2>(), g.ckx_base.as<int64_t>(),
                                    g.pair_ring.as<int2>(), g.ls.as<int>(), g.st64.as<double2>(), g.y64.as<double>(),
                                    (double2*)F, fs, L, g.npair, R, nm, stall_of(g));
  CMBWS_LAUNCH_CHECK();
  return CMBWS_OK;
}

template <int NM>
int launch_synth(int nm, const Grid& g, const void* alm, int64_t as, void* F, int64_t fs, cudaStream_t s) {
  int v = 1;
  if (autotune_mode() != 0)
    CMBWS_TRY(autotune_pick(
        g, synth_tune_key(CMBWS_FP64, NM), kFxTiles, 1,
        [&](int vv) { return launch_synth_variant<NM>(vv, nm, g, alm, as, F, fs, s); }, s, &v));
  return launch_synth_variant<NM>(v, nm, g, alm, as, F, fs, s);
}

// ---- adjoint ----
constexpr int kAdjK = 32;                       // ring pairs per stage (two K steps)
constexpr int kAdjTile = kM * kAdjK * 2;        // one digit of A
constexpr int kAdjOct = kAdjK * 16;             // bytes between rows 8 i and 8 (i + 1) of A
template <typename C>
struct AdjLayout {
  static constexpr int kA = 0;
  static constexpr int kB = kFxDig * kAdjTile;       // B of a stage (two K steps)
  static constexpr int kCoef = kB + 2 * C::kBStep;   // int4[128]
  static constexpr int kCorr = kCoef + kM * 16;      // fxu_t[2 W][2]
  static constexpr int kBar = kCorr + 2 * C::W * 16; // uint64_t[2]
  static constexpr int kMisc = kBar + 16;            // tensor memory base, bad flag
  static constexpr int kBytes = kMisc + 16;
};

__device__ __forceinline__ unsigned part_exp(double v) {
  return ((unsigned)__double2hiint(v) >> 20) & 0x7ffu;
}

// ee[map][m] = exponent bound of the map's ring parts e 2^-S at m, S the scale of their pair (fixed.h):
// |e 2^-S| < 2^ee (kNotFinite: not all finite).  The ring parts become fixed point at that scale in place
// (zeros if not finite, and for pairs that never start), once for all tiles of l.  Without the pair's
// scale, a bright ring at a pole, whose Legendre values at high m are all small, would set ee there: one
// pixel of 1e10 over unit noise in the first ring of a GL grid with L = 63 left an m with errors of 4e-9
// of its largest coefficient; 3e-14 with it, as from FP64 arithmetic.
constexpr int kNotFinite = 1 << 20;
template <int NM>
__global__ void __launch_bounds__(256)
k_eo_fix(double* __restrict__ eo, int npair, int L, const uint8_t* __restrict__ sx, int* __restrict__ ee,
         int nmaps) {
  const int nm = NM <= 4 ? NM : nmaps;
  __shared__ int s_e[NM];
  const int m = blockIdx.x, tid = threadIdx.x;
  if (tid < NM) s_e[tid] = -kNotFinite;
  __syncthreads();
  double* src = eo + (int64_t)m * npair * 4 * nm;
  const uint8_t* sm = sx + (int64_t)m * npair;
  int e[NM];
#pragma unroll
  for (int k = 0; k < NM; ++k) e[k] = -kNotFinite;
  for (int i = tid; i < 2 * npair; i += 256) {  // (pair, parity): 2 nm values
    const double2* v = reinterpret_cast<const double2*>(src) + (int64_t)i * nm;
    const int S = sm[i >> 1];
#pragma unroll
    for (int k = 0; k < NM; ++k)
      if (k < nm) {
        const int x = (int)max(part_exp(v[k].x), part_exp(v[k].y));
        if (x == 0x7ff) e[k] = kNotFinite;
        else if (S) e[k] = max(e[k], x - 1022 - S);
      }
  }
#pragma unroll
  for (int k = 0; k < NM; ++k) {
    const int v = __reduce_max_sync(kFull, e[k]);
    if ((tid & 31) == 0) atomicMax(&s_e[k], v);
  }
  __syncthreads();
  if (tid < nm) ee[(int64_t)tid * (L + 1) + m] = s_e[tid];
  int sc[NM];
#pragma unroll
  for (int k = 0; k < NM; ++k) sc[k] = s_e[k];
  for (int i = tid; i < 2 * npair; i += 256) {
    double2* v = reinterpret_cast<double2*>(src) + (int64_t)i * nm;
    const int S = sm[i >> 1];
#pragma unroll
    for (int k = 0; k < NM; ++k)
      if (k < nm) {
        const bool ok = S && sc[k] < kNotFinite;
        const int x = kFxABits - sc[k] - S;
        const double2 d = v[k];
        v[k] = make_double2(__longlong_as_double(ok ? fx_from_double(d.x, x) : 0),
                            __longlong_as_double(ok ? fx_from_double(d.y, x) : 0));
      }
  }
}

// One CTA per (m, 128 values of l) loops over the ring pairs, 32 per stage: lane = pair, warp =
// chunk of 16 values of l, which each thread walks from the chunk's checkpoint; rows of A are
// values of l (MN-major: a thread writes 8 consecutive values of its pair as one 16-byte row).
// Every output has one owner; stages without a started pair are skipped.
// One buffer of B, filled once the previous stage's MMAs are done: a second one would leave room for two
// CTAs per SM only.  Bound as the synthesis is (tensor pipe 17 %).  Against the FP64 pipe, Nside 1024, 3
// maps: 107.9 -> 19.5 ms with k_eo_fix (18.1 with 7 digits and two buffers); GL L = 1000, 1 map: 1.77 ->
// 0.64 ms.
template <int NM>
__global__ void __launch_bounds__(kNT, Cols<NM>::kCtas)
k_leg_adj_fx(const fx_t* __restrict__ eo, const int* __restrict__ ee, const double* __restrict__ Acoef,
             const int* __restrict__ ls_tab, const ulonglong2* __restrict__ st, const uint64_t* __restrict__ xfx,
             const ulonglong2* __restrict__ ck, const int64_t* __restrict__ ck_base,
             const int* __restrict__ tmin, const double* __restrict__ c64, double2* __restrict__ out,
             int64_t nlm, int L, int npair, int nmaps, long long stall) {
  using C = Cols<NM>;
  using LY = AdjLayout<C>;
  constexpr int W = C::W;
  const int nm = NM <= 4 ? NM : nmaps, P = 2 * nm;
  static_assert(kFxChunk == 16 && kAdjK == 32 && kTileMinPT == 16, "stage shape");
  const int m = blockIdx.y;
  const int lb0 = m + kM * (int)blockIdx.x;  // first l of the tile
  if (lb0 > L) return;                       // CTA-uniform, before any barrier
  extern __shared__ __align__(1024) unsigned char sm[];
  int4* s_coef = reinterpret_cast<int4*>(sm + LY::kCoef);
  fxu_t* s_corr = reinterpret_cast<fxu_t*>(sm + LY::kCorr);
  uint64_t* mbar = reinterpret_cast<uint64_t*>(sm + LY::kBar);
  uint32_t* s_tb = reinterpret_cast<uint32_t*>(sm + LY::kMisc);
  int* s_bad = reinterpret_cast<int*>(sm + LY::kMisc + 4);

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int64_t lmo = lm_off(L, m) - m;
  const int llast = min(L, lb0 + kM - 1);
  const int ntm = (npair + kTileMinPT - 1) / kTileMinPT;
  const int nst = (npair + kAdjK - 1) / kAdjK;
  const int* tm = tmin + (int64_t)m * ntm;
  // first stage from s on with a pair that starts by the tile's last l
  auto next_stage = [&](int s) {
    while (s < nst && tm[2 * s] > llast && (2 * s + 1 >= ntm || tm[2 * s + 1] > llast)) ++s;
    return s;
  };
  int s = next_stage(0);
  if (s >= nst) {  // no pair has a significant value in the tile: the sums are zero
    const int l = lb0 + tid;
    if (tid < kM && l <= L)
      for (int k = 0; k < nm; ++k) out[k * nlm + lmo + l] = make_double2(0.0, 0.0);
    return;
  }
  if (tid == 0) {
    *s_bad = 0;
    mbar_init(&mbar[0], 1);
    mbar_init(&mbar[1], 1);
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  }
  if (tid < 4 * W) s_corr[tid] = 0;
  if (tid < kM) {
    const int l = lb0 + tid;
    s_coef[tid] = fx_coef(l <= L ? Acoef[lmo + l] : 0.0);
  }
  for (int i = tid; i < 2 * C::kBStep / 16; i += kNT)  // B columns of absent maps stay zero
    reinterpret_cast<uint4*>(sm + LY::kB)[i] = make_uint4(0, 0, 0, 0);
  if (stall > 0 && tid == 0 && !mbar_wait(&mbar[1], 0, stall)) *s_bad = 1;
  __syncwarp();
  if (warp == 0) tmem_alloc<C::kTmem>(s_tb);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tb = *s_tb;
  const uint32_t lane_base = (uint32_t)((warp & 3) * 32) << 16;

  // chunk of this warp
  const int l0 = lb0 + kFxChunk * warp;
  const bool cval = l0 <= L;
  const int nck = (L - m + kFxChunk) / kFxChunk;
  const ulonglong2* ckc = ck + (cval ? ck_base[m] + (l0 - m) / kFxChunk : 0);  // + p * nck
  const int* lsm = ls_tab + (int64_t)m * npair;
  const ulonglong2* stm = st + (int64_t)m * npair;
  unsigned char* arow = sm + LY::kA + 2 * warp * kAdjOct + lane * 16;

  // this thread's ring parts of a stage: column nn of parity par, kPP pairs from 8 oct + kPP sub on
  constexpr int kPP = W / 4, kSub = 8 / kPP;
  const int sub = tid & (kSub - 1), nn = (tid / kSub) & (W - 1), oct = (tid >> 5) & 3, par = tid >> 7;
  const int col = (nn & 1) * (W / 2) + (nn >> 1);
  const bool bon = nn < P;
  const fx_t* bsrc = eo + (int64_t)m * npair * 2 * P + par * P + nn;
  unsigned char* bdst = sm + LY::kB + (oct >> 1) * C::kBStep + par * W * 32 + (oct & 1) * 128 +
                        (col >> 3) * 256 + (col & 7) * 16 + sub * kPP * 2;

  // inputs of a stage, loaded one stage ahead
  struct In {
    fx_t e[kPP];
    ulonglong2 c;
    uint64_t x;
    int ls;
  };
  auto load = [&](int t, In& in) {
    const int p = t * kAdjK + lane;
    const bool ok = t < nst && p < npair;
    in.ls = ok ? lsm[p] : INT_MAX;
    in.x = ok ? xfx[p] : 0;
    in.c = make_ulonglong2(0, 0);
    if (ok && cval) in.c = ckc[(int64_t)p * nck];
#pragma unroll
    for (int i = 0; i < kPP; ++i) {
      const int q = t * kAdjK + 8 * oct + kPP * sub + i;
      in.e[i] = 0;
      if (bon && t < nst && q < npair) in.e[i] = bsrc[(int64_t)q * 2 * P];
    }
  };
  In in;
  load(s, in);

  const int grp = tid >> 7;  // real (0) or imaginary (1) parts of row tid mod 128
  FxSum acc[NM];
  fx_t shi = 0, slo = 0;
  bool bad = false, zeroed = false;
  for (int k = 0; s < nst; ++k) {
    const int sn = next_stage(s + 1);
    const int p = s * kAdjK + lane, ls = in.ls;
    const unsigned xh = (unsigned)(in.x >> 32), xl = (unsigned)in.x;
    const bool on = cval && __any_sync(kFull, ls <= min(L, l0 + kFxChunk - 1));
    FxState w, s0;
    if (on) {
      w = fx_unpack(in.c);  // zeros if the pair starts later
      const bool inj = ls > l0 && ls < l0 + kFxChunk && ls <= L;
      if (__any_sync(kFull, inj)) {
        if (inj) s0 = fx_unpack(stm[p]);
        if ((ls - m) & 2) fx_negate(s0);
      }
    }
    fx_t ev[kPP];
#pragma unroll
    for (int i = 0; i < kPP; ++i) ev[i] = in.e[i];
    load(sn, in);
    auto wait = [&]() {  // the previous stage's MMAs have read the tile
      if (k >= 1 && !*s_bad && !mbar_wait(&mbar[0], (k - 1) & 1)) bad = true;
    };
    if (on) {
      const int lst = ls > l0 ? ls : INT_MAX;
#pragma unroll 1
      for (int h = 0; h < 2; ++h)
        fx_walk8(w, s_coef + kFxChunk * warp + 8 * h, xh, xl, l0 + 8 * h, lst, s0, h == 0,
                 arow + h * kAdjOct, kAdjTile, wait);
      zeroed = false;
    } else {
      wait();
      if (!zeroed)  // no pair of the stage has started in this chunk: zero digits
#pragma unroll
        for (int i = 0; i < kFxDig; ++i) {
          const unsigned z = zero_digit(i);
#pragma unroll
          for (int h = 0; h < 2; ++h)
            *reinterpret_cast<uint4*>(arow + i * kAdjTile + h * kAdjOct) = make_uint4(z, z, z, z);
        }
      zeroed = true;
    }
    if (bon) {  // B of this stage: the previous one was waited for
#pragma unroll
      for (int i = 0; i < kPP; i += 2) {
        const fx_t v = ev[i], u = ev[i + 1];
        shi += (v >> 30) + (u >> 30);
        slo += (v & ((1 << 30) - 1)) + (u & ((1 << 30) - 1));
        unsigned dig[kFxDig];
        fx_coef_digits(v, u, dig);
#pragma unroll
        for (int j = 0; j < kFxDig; ++j)
          *reinterpret_cast<unsigned*>(bdst + j * C::kDig + 2 * i) = dig[j];
      }
    }
    fence_smem_async();
    tc_fence_before();
    if (bad) atomicOr(s_bad, 1);
    __syncthreads();
    const bool first = (k & 1) == 0;  // sums are read after every second stage (64 pairs)
    if (tid == 0 && !*s_bad) {
      tc_fence_after();
#pragma unroll
      for (int ks = 0; ks < 2; ++ks)
        mma_step<C>(tb, smem_addr(sm + LY::kA) + ks * 256, kAdjTile, 128, kAdjOct,
                 smem_addr(sm + LY::kB + ks * C::kBStep), true, first && ks == 0);
      tc_commit(&mbar[0]);
    }
    if ((k & 1) == 1 || sn >= nst) {
      if (!*s_bad && !mbar_wait(&mbar[0], k & 1)) bad = true;
      tc_fence_after();
      int prev[NM];
      const int odd = tid & 1;  // parity of l - m of this thread's row
#pragma unroll
      for (int b = 0; b < kFxBlk; ++b) {
        uint32_t d[W / 2], f[W / 2];
        const uint32_t c = tb + lane_base + 2 * W * b + grp * (W / 2);
        tmem_ld<W / 2>(c, d);
        tmem_ld<W / 2>(c + W, f);
        tmem_ld_wait();
#pragma unroll
        for (int q = 0; q < NM; ++q) acc[q].add(b, digit_sum(odd ? f[q] : d[q]), prev[q]);
      }
      tc_fence_before();  // read before the next stage's MMAs, which follow its barrier
    }
    s = sn;
  }
  if (bon) {
    atomicAdd(&s_corr[2 * (par * W + nn)], (fxu_t)shi);
    atomicAdd(&s_corr[2 * (par * W + nn) + 1], (fxu_t)slo);
  }
  if (bad) atomicOr(s_bad, 1);
  __syncthreads();
  const bool failed = *s_bad != 0;
  if (tid == 0 && failed) atomicOr(&g_fx_status, 1u);
  if (warp == 0) tmem_free<C::kTmem>(tb);
  const int l = lb0 + (tid & (kM - 1));  // row of D
  if (l > L) return;
  const fxu_t* corr = s_corr + 2 * W * (tid & 1) + 2 * grp;
  // sigma of l, and the ring FFT's sqrt(2)
  const double cc = ((tid & 2) ? -c64[lmo + l] : c64[lmo + l]) * (m > 0 ? 1.41421356237309504880 : 1.0);
  double* o = reinterpret_cast<double*>(out + lmo + l) + grp;
#pragma unroll
  for (int q = 0; q < NM; ++q) {
    if (q >= nm) break;
    const int ea = ee[(int64_t)q * (L + 1) + m];
    const double v = acc[q].value((fx_t)corr[4 * q], (fx_t)corr[4 * q + 1], ea - 6);
    // a map with a non-finite ring part, and a timed-out wait, give NaN
    o[2 * q * nlm] = (failed || ea == kNotFinite) ? fx_nan() : cc * v;
  }
}

template <int NM>
int launch_adj(int nm, const Grid& g, double* eo, int* ee, double* out, cudaStream_t s) {
  using LY = AdjLayout<Cols<NM>>;
  const int L = g.lmax;
  ProfScope ps(PROF_LEG_ADJ, s, 1, leg_work(g, nm));
  k_eo_fix<NM><<<L + 1, 256, 0, s>>>(eo, g.npair, L, g.sx.as<uint8_t>(), ee, nm);
  CMBWS_LAUNCH_CHECK();
  dim3 grd((L + kM) / kM, L + 1);
  auto kern = k_leg_adj_fx<NM>;
  CMBWS_TRY(ensure_dyn_smem((const void*)kern, LY::kBytes));
  kern<<<grd, kNT, LY::kBytes, s>>>(reinterpret_cast<const fx_t*>(eo), ee, g.A64.as<double>(), g.lsx.as<int>(),
                                    g.stx.as<ulonglong2>(), g.xfx.as<uint64_t>(), g.ckx.as<ulonglong2>(),
                                    g.ckx_base.as<int64_t>(), g.lsx_tmin.as<int>(), g.c64.as<double>(),
                                    (double2*)out, nlm_of(L), L, g.npair, nm, stall_of(g));
  CMBWS_LAUNCH_CHECK();
  return CMBWS_OK;
}

}  // namespace

int legendre_synth_fx(const Grid& g, int nmaps, const void* alm, void* F, cudaStream_t s) {
  CMBWS_TRY(grid_ensure_fx(g, s));
  const int64_t as = nlm_of(g.lmax), fs = (int64_t)g.nring * (g.lmax + 1);
  for (int k0 = 0; k0 < nmaps; k0 += kFxMaps) {
    const int nm = nmaps - k0 < kFxMaps ? nmaps - k0 : kFxMaps;
    const void* a = (const double2*)alm + k0 * as;
    void* f = (double2*)F + k0 * fs;
    switch (nm) {
      case 1: CMBWS_TRY(launch_synth<1>(nm, g, a, as, f, fs, s)); break;
      case 2: CMBWS_TRY(launch_synth<2>(nm, g, a, as, f, fs, s)); break;
      case 3: CMBWS_TRY(launch_synth<3>(nm, g, a, as, f, fs, s)); break;
      case 4: CMBWS_TRY(launch_synth<4>(nm, g, a, as, f, fs, s)); break;
      case 5:
      case 6: CMBWS_TRY(launch_synth<6>(nm, g, a, as, f, fs, s)); break;
      default: CMBWS_TRY(launch_synth<8>(nm, g, a, as, f, fs, s)); break;
    }
  }
  return CMBWS_OK;
}

int legendre_adjoint_fx(const Grid& g, int nmaps, void* eo, int* ee, double* out, cudaStream_t s) {
  CMBWS_TRY(grid_ensure_fx(g, s));
  const int64_t nlm = nlm_of(g.lmax), cs = (int64_t)(g.lmax + 1) * g.npair * 4;
  for (int k0 = 0; k0 < nmaps; k0 += kFxMaps) {
    const int nm = nmaps - k0 < kFxMaps ? nmaps - k0 : kFxMaps;
    double* e = (double*)eo + k0 * cs;
    int* x = ee + (int64_t)k0 * (g.lmax + 1);
    double* o = out + 2 * k0 * nlm;
    switch (nm) {
      case 1: CMBWS_TRY(launch_adj<1>(nm, g, e, x, o, s)); break;
      case 2: CMBWS_TRY(launch_adj<2>(nm, g, e, x, o, s)); break;
      case 3: CMBWS_TRY(launch_adj<3>(nm, g, e, x, o, s)); break;
      case 4: CMBWS_TRY(launch_adj<4>(nm, g, e, x, o, s)); break;
      case 5:
      case 6: CMBWS_TRY(launch_adj<6>(nm, g, e, x, o, s)); break;
      default: CMBWS_TRY(launch_adj<8>(nm, g, e, x, o, s)); break;
    }
  }
  return CMBWS_OK;
}

int fx_stall_waits(long long cycles) {
  int dev = 0;
  CMBWS_CUDA(cudaGetDevice(&dev));
  if (dev < kMaxDevices) g_stall[dev].store(cycles, std::memory_order_relaxed);
  return CMBWS_OK;
}

int fx_status_take(bool* timed_out) {
  unsigned int v = 0;
  CMBWS_CUDA(cudaMemcpyFromSymbol(&v, g_fx_status, sizeof(v)));
  *timed_out = (v & 1u) != 0;
  if (v) {
    const unsigned int zero = 0;
    CMBWS_CUDA(cudaMemcpyToSymbol(g_fx_status, &zero, sizeof(zero)));
  }
  return CMBWS_OK;
}

}  // namespace cmbws
