// Associated-Legendre stage of the spherical harmonic transform (Sec. 2.1),
// the dominant cost of every apply of A and M_PI (Sec. 3.3 counts SHTs).
//
// Synthesis, per m and ring pair (theta, pi - theta):
//   F_m(theta) = sum_l lambda_lm(theta) a_lm,  with lambda_lm(pi - theta) = (-1)^(l+m) lambda_lm(theta),
// so E = sum over l+m even and O = sum over l+m odd give F_north = E + O and
// F_south = E - O from one recurrence.  Adjoint synthesis is the transpose:
//   a_lm = sum_pairs lambda_lm(theta) (E-part or O-part of the ring spectra).
//
// FP32 on the CUDA cores (the recurrence costs two operations per (l, m, pair), the contraction
// two FMAs per map); the FP64 stage is in legendre_fx.cu, the double-float one in
// legendre_df.cu, the TF32 and BF16 ones in legendre_tc.cu.
// * synthesis: one CTA per (m, block of ring pairs); each thread owns R pairs, walks l
//   upwards two steps at a time (even/odd partners) and starts each pair at
//   its precomputed first significant l (start values injected there); the coefficients of the
//   current l-chunk are staged in shared memory and read as broadcasts; every map of the grid
//   group shares one recurrence (NM maps per launch);
// * adjoint: one thread per chunk of l, which restarts every pair's recurrence from stored
//   checkpoints (k_leg_adj_ck below).
#include <climits>

#include "common.h"

namespace cmbws {

namespace {

constexpr unsigned kFull = 0xffffffffu;

template <int NM, int R, int NT, int CH>
__global__ void __launch_bounds__(NT)
k_leg_synth(const float2* __restrict__ alm, int64_t alm_stride,
            const float* __restrict__ Acoef, const float* __restrict__ brs,
            const int* __restrict__ ls_tab,
            const float2* __restrict__ st, const float* __restrict__ yr,
            const int2* __restrict__ pring, float2* __restrict__ F, int64_t F_stride,
            int L, int npair, int nring) {
  __shared__ __align__(16) float sA[CH];
  __shared__ __align__(16) float2 sa[NM][CH];
  __shared__ __align__(16) float sBRS[3][CH];  // difference form
  __shared__ int s_lo;

  const int m = blockIdx.y;
  const int64_t lmo = lm_off(L, m) - m;  // index of (m, l) is lmo + l
  const int pbase = blockIdx.x * NT * R + threadIdx.x;

  int ls[R];
  float y[R], mu1[R], mu2[R];
  float2 inj[R];
  float eR[R][NM], eI[R][NM], oR[R][NM], oI[R][NM];
  int mylo = INT_MAX;
#pragma unroll
  for (int i = 0; i < R; ++i) {
    const int p = pbase + i * NT;
    if (p < npair) {
      ls[i] = ls_tab[(int64_t)m * npair + p];
      y[i] = yr[p];
      inj[i] = st[(int64_t)m * npair + p];
    } else {
      ls[i] = INT_MAX;
      y[i] = 0;
      inj[i].x = inj[i].y = 0;
    }
    mylo = min(mylo, ls[i]);
    mu1[i] = mu2[i] = 0;
#pragma unroll
    for (int k = 0; k < NM; ++k) eR[i][k] = eI[i][k] = oR[i][k] = oI[i][k] = 0;
  }
  if (threadIdx.x == 0) s_lo = INT_MAX;
  __syncthreads();
  atomicMin(&s_lo, mylo);
  __syncthreads();
  const int lo = s_lo;
  int nxt = mylo;  // next l at which one of this thread's pairs starts
  // first l at which a pair of this warp starts: the warp skips every chunk before it (its
  // recurrence values are zero there; warps without a valid pair skip all chunks)
  const int wlo = __reduce_min_sync(kFull, mylo);
  // warps holding a polar ring pair run the difference form (warp-uniform)
  bool mine = false;
#pragma unroll
  for (int i = 0; i < R; ++i) mine |= (pbase + i * NT < npair) && y[i] < kPolarY;
  const bool polar = __any_sync(kFull, mine);

  for (int c0 = lo; c0 <= L; c0 += CH) {
    __syncthreads();
    for (int j = threadIdx.x; j < CH; j += NT) {
      const int l = c0 + j;
      const bool ok = l <= L;
      sA[j] = ok ? Acoef[lmo + l] : 0.f;
#pragma unroll
      for (int q = 0; q < 3; ++q) sBRS[q][j] = ok ? brs[3 * (lmo + l) + q] : 0.f;
#pragma unroll
      for (int k = 0; k < NM; ++k) {
        float2 v = make_float2(0.f, 0.f);
        if (ok) v = alm[k * alm_stride + lmo + l];
        sa[k][j] = v;
      }
    }
    __syncthreads();
    // values of l in this chunk (the last chunk stops at L; an even count, the partner of
    // an odd tail reads the zeros staged beyond L)
    const int jn = min(CH, (L - c0 + 2) & ~1);
    if (c0 + jn <= wlo) continue;
    if (polar) {
      // mu2 holds e_{l-1} = mu_{l-1} - R_{l-1} mu_{l-2} in this form
#pragma unroll 2
      for (int j = 0; j < jn; j += 2) {
        const int l = c0 + j;
        const float A0 = sA[j], A1 = sA[j + 1];
        const float B0 = sBRS[0][j], B1 = sBRS[0][j + 1], R0 = sBRS[1][j], R1 = sBRS[1][j + 1];
        const float S0 = sBRS[2][j], S1 = sBRS[2][j + 1];
        float ma[R], mb[R];
#pragma unroll
        for (int i = 0; i < R; ++i) {
          float e = fmaf(fmaf(-A0, y[i], B0), mu1[i], S0 * mu2[i]);
          ma[i] = fmaf(R0, mu1[i], e);
          e = fmaf(fmaf(-A1, y[i], B1), ma[i], S1 * e);
          mb[i] = fmaf(R1, ma[i], e);
          mu2[i] = e;
        }
        if (l == nxt) {
          int nn = INT_MAX;
#pragma unroll
          for (int i = 0; i < R; ++i) {
            if (ls[i] == l) {
              ma[i] = inj[i].x;
              mb[i] = inj[i].y;
              mu2[i] = fmaf(-R1, inj[i].x, inj[i].y);
            }
            if (ls[i] > l) nn = min(nn, ls[i]);
          }
          nxt = nn;
        }
#pragma unroll
        for (int i = 0; i < R; ++i) mu1[i] = mb[i];
#pragma unroll
        for (int k = 0; k < NM; ++k) {
          const float2 a0 = sa[k][j], a1 = sa[k][j + 1];
#pragma unroll
          for (int i = 0; i < R; ++i) {
            eR[i][k] += ma[i] * a0.x;
            eI[i][k] += ma[i] * a0.y;
            oR[i][k] += mb[i] * a1.x;
            oI[i][k] += mb[i] * a1.y;
          }
        }
      }
      continue;
    }
#pragma unroll 2
    for (int j = 0; j < jn; j += 2) {
      const int l = c0 + j;
      const float A0 = sA[j], A1 = sA[j + 1];
      float ma[R], mb[R];
#pragma unroll
      for (int i = 0; i < R; ++i) {
        ma[i] = fma(-A0, y[i], A0) * mu1[i] - mu2[i];
        mb[i] = fma(-A1, y[i], A1) * ma[i] - mu1[i];
      }
      if (l == nxt) {
        int nn = INT_MAX;
#pragma unroll
        for (int i = 0; i < R; ++i) {
          if (ls[i] == l) {
            ma[i] = inj[i].x;
            mb[i] = inj[i].y;
          }
          if (ls[i] > l) nn = min(nn, ls[i]);
        }
        nxt = nn;
      }
#pragma unroll
      for (int i = 0; i < R; ++i) {
        mu2[i] = ma[i];
        mu1[i] = mb[i];
      }
#pragma unroll
      for (int k = 0; k < NM; ++k) {
        const float2 a0 = sa[k][j], a1 = sa[k][j + 1];
#pragma unroll
        for (int i = 0; i < R; ++i) {
          eR[i][k] += ma[i] * a0.x;
          eI[i][k] += ma[i] * a0.y;
          oR[i][k] += mb[i] * a1.x;
          oI[i][k] += mb[i] * a1.y;
        }
      }
    }
  }

#pragma unroll
  for (int i = 0; i < R; ++i) {
    const int p = pbase + i * NT;
    if (p >= npair) continue;
    const int2 rr = pring[p];
#pragma unroll
    for (int k = 0; k < NM; ++k) {
      float2 fn, fs;
      fn.x = eR[i][k] + oR[i][k];
      fn.y = eI[i][k] + oI[i][k];
      F[k * F_stride + (int64_t)rr.x * (L + 1) + m] = fn;
      if (rr.y >= 0) {
        fs.x = eR[i][k] - oR[i][k];
        fs.y = eI[i][k] - oI[i][k];
        F[k * F_stride + (int64_t)rr.y * (L + 1) + m] = fs;
      }
    }
  }
}

// FP32 adjoint from chunk checkpoints: one thread per chunk of kChunk values of l
// (a CTA covers NT consecutive chunks of one m) loops over every ring pair of the
// grid.  Each pair's recurrence restarts at the chunk from the stored FP64-computed
// values (setup.cu), so no thread needs another thread's sums: each output (l, m) is
// owned by one thread and summed over the pairs in a fixed order.
// Tiles of PT pairs are staged in shared memory with cp.async, double-buffered: the
// per-pair even/odd parts E, O (written by the forward ring FFT), y, the start index and values,
// and each thread's own column of checkpoints, so the HBM reads of the next tile
// overlap the arithmetic of the current one.
// E/O parts of every (pair, m): eo[(m * npair + p) * 2P + q], q < P even-l parts (north +
// south), q >= P odd-l parts (north - south), parts = (re, im) per map.
template <int NM, int PT>
struct AdjCkWarp {  // one warp's double-buffered tile
  float eo[2][PT][4 * NM];
  float y[2][PT];
  int ls[2][PT];
  float2 st[2][PT];
  float2 ck[2][PT][32];
};

template <int NM, int NT, int PT>
__global__ void __launch_bounds__(NT)
k_leg_adj_ck(const float* __restrict__ eo, const float* __restrict__ Acoef,
             const int* __restrict__ ls_tab, const float2* __restrict__ st,
             const float* __restrict__ yr, const float2* __restrict__ ck,
             const int64_t* __restrict__ ck_base, const int2* __restrict__ tasks, int ntask,
             const int* __restrict__ tmin, const double* __restrict__ c64,
             double2* __restrict__ out, int64_t nlm, int L, int npair) {
  static_assert(PT == kTileMinPT, "the tile-start table is built for kTileMinPT pairs per tile");
  constexpr int P = 2 * NM;
  constexpr int K = kChunk;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  AdjCkWarp<NM, PT>& S = reinterpret_cast<AdjCkWarp<NM, PT>*>(smem_raw)[warp];
  // every warp takes one task (32 consecutive chunks of one m); warps of a CTA are independent
  const int task = blockIdx.x * (NT / 32) + warp;
  if (task >= ntask) return;  // warp-uniform: no block barrier below
  const int2 tk = tasks[task];
  const int m = tk.x;
  const int nck = (L - m + K) / K;
  const int cw = tk.y;  // first chunk of this warp
  const int c = cw + lane;
  const bool valid = c < nck;
  const int l0 = m + K * c;
  const int64_t lmo = lm_off(L, m) - m;
  float Al[K];
#pragma unroll
  for (int j = 0; j < K; ++j) Al[j] = (valid && l0 + j <= L) ? Acoef[lmo + l0 + j] : 0.f;
  float acc[K][P];
#pragma unroll
  for (int j = 0; j < K; ++j)
#pragma unroll
    for (int q = 0; q < P; ++q) acc[j][q] = 0.f;
  const float2* ckc = ck + ck_base[m] + c;  // + p * nck
  const float* eom = eo + (int64_t)m * npair * 2 * P;
  const int ntile = (npair + PT - 1) / PT;
  // Pairs are not sorted by start; a tile whose pairs all start after the warp's last l
  // (tmin, the smallest start of the tile) adds nothing to this warp's outputs and is not
  // staged.  Pairs of a visited tile that have not started are skipped one by one.
  const int llast = min(L, m + K * (cw + 32) - 1);
  const int* tm = tmin + (int64_t)m * ntile;
  auto next_tile = [&](int t) {
    while (t < ntile && tm[t] > llast) ++t;
    return t;
  };

  auto stage = [&](int t, int bf) {
    const int p0 = t * PT;
    const int np = min(PT, npair - p0);
    const float* src = eom + (int64_t)p0 * 2 * P;
    for (int i = lane; i < np * NM; i += 32) cp_async16(&S.eo[bf][0][0] + 4 * i, src + 4 * i);
    for (int i = lane; i < np; i += 32) {
      cp_async4(&S.y[bf][i], yr + p0 + i);
      cp_async4(&S.ls[bf][i], ls_tab + (int64_t)m * npair + p0 + i);
      cp_async8(&S.st[bf][i], st + (int64_t)m * npair + p0 + i);
    }
    if (valid)
      for (int i = 0; i < np; ++i) cp_async8(&S.ck[bf][i][lane], ckc + (int64_t)(p0 + i) * nck);
    cp_async_commit();
  };

  int t = next_tile(0);
  if (t < ntile) stage(t, 0);
  for (int k = 0; t < ntile; ++k) {
    const int tn = next_tile(t + 1);
    if (tn < ntile) {
      stage(tn, (k + 1) & 1);
      cp_async_wait<1>();
    } else {
      cp_async_wait<0>();
    }
    __syncwarp();
    if (valid) {
      const int bf = k & 1;
      const int np = min(PT, npair - t * PT);
      for (int i = 0; i < np; ++i) {
        const int lsp = S.ls[bf][i];
        if (lsp > l0 + K - 1) continue;  // the pair starts after this chunk
        const float2 cv = S.ck[bf][i][lane];
        float ma = cv.x, mb = cv.y;
        if (lsp == l0) {
          ma = S.st[bf][i].x;
          mb = S.st[bf][i].y;
        }
        const float yv = S.y[bf][i];
        const float* e = S.eo[bf][i];
#pragma unroll
        for (int q = 0; q < P; ++q) {
          acc[0][q] += ma * e[q];
          acc[1][q] += mb * e[P + q];
        }
#pragma unroll
        for (int j = 2; j < K; j += 2) {
          float na = fmaf(-Al[j], yv, Al[j]) * mb - ma;
          float nb = fmaf(-Al[j + 1], yv, Al[j + 1]) * na - mb;
          if (l0 + j == lsp) {
            na = S.st[bf][i].x;
            nb = S.st[bf][i].y;
          }
          ma = na;
          mb = nb;
#pragma unroll
          for (int q = 0; q < P; ++q) {
            acc[j][q] += ma * e[q];
            acc[j + 1][q] += mb * e[P + q];
          }
        }
      }
    }
    __syncwarp();  // buffer k & 1 is restaged two iterations later
    t = tn;
  }
  if (!valid) return;
#pragma unroll
  for (int j = 0; j < K; ++j) {
    const int l = l0 + j;
    if (l > L) break;
    const int64_t i = lmo + l;
    const double cc = c64[i];
#pragma unroll
    for (int k = 0; k < NM; ++k)
      out[k * nlm + i] = make_double2(cc * (double)acc[j][2 * k], cc * (double)acc[j][2 * k + 1]);
  }
}

constexpr int kSynthCH = 256;  // values of l staged at once

template <int NM, int R, int NT>
int launch_synth_rn(const Grid& g, const void* alm, int64_t alm_stride, void* F, int64_t F_stride,
                    cudaStream_t s) {
  const int L = g.lmax;
  dim3 grd((g.npair + NT * R - 1) / (NT * R), L + 1);
  ProfScope ps(PROF_LEG_SYNTH, s, 0, leg_work(g, NM));
  k_leg_synth<NM, R, NT, kSynthCH><<<grd, NT, 0, s>>>(
      (const float2*)alm, alm_stride, g.A32.as<float>(), g.BRS32.as<float>(), g.ls.as<int>(),
      g.st32.as<float2>(), g.y32.as<float>(), g.pair_ring.as<int2>(), (float2*)F, F_stride, L,
      g.npair, g.nring);
  CMBWS_LAUNCH_CHECK();
  return CMBWS_OK;
}

// Tile variants of the synthesis (ring pairs per thread R, threads per CTA NT): variant 0 is
// the default for large grids; the others trade pairs per CTA (fewer idle lanes on grids
// with few ring pairs) against coefficient reuse (R = 4: a shared-memory broadcast serves
// four recurrences).  The autotuner picks one per (grid, precision, maps).
constexpr int kSynthVariants = 4;

template <int NM>
int launch_synth_variant(int v, const Grid& g, const void* alm, int64_t as, void* F, int64_t fs,
                         cudaStream_t s) {
  switch (v) {
    case 1: return launch_synth_rn<NM, 1, 128>(g, alm, as, F, fs, s);
    case 2: return launch_synth_rn<NM, 1, 64>(g, alm, as, F, fs, s);
    case 3: return launch_synth_rn<NM, 4, 64>(g, alm, as, F, fs, s);
    default: return launch_synth_rn<NM, 2, 128>(g, alm, as, F, fs, s);
  }
}

// heuristic: the smallest CTA (in ring pairs) that holds all pairs of the grid
inline int synth_heuristic(const Grid& g) { return g.npair <= 64 ? 2 : g.npair <= 128 ? 1 : 0; }

template <int NM>
int launch_synth(const Grid& g, const void* alm, int64_t as, void* F, int64_t fs, cudaStream_t s) {
  int v = 0;
  CMBWS_TRY(autotune_pick(g, synth_tune_key(CMBWS_FP32, NM), kSynthVariants, synth_heuristic(g),
                          [&](int vv) { return launch_synth_variant<NM>(vv, g, alm, as, F, fs, s); },
                          s, &v));
  return launch_synth_variant<NM>(v, g, alm, as, F, fs, s);
}

template <int NM>
int launch_adj_ck(const Grid& g, const float* eo, double* out, cudaStream_t s) {
  // one warp per CTA: the warps are independent tasks (no CTA barrier), so an SM holds as
  // many as its registers allow (16 at 120 registers) instead of whole 4-warp CTAs (12 at 130):
  // 3.29 against 3.77 ms per Nside-1024 launch of 3 maps
  constexpr int NT = 32, PT = 16;
  const int L = g.lmax;
  const int64_t nlm = nlm_of(L);
  dim3 grd((g.nwt32 + NT / 32 - 1) / (NT / 32));
  constexpr size_t sm = sizeof(AdjCkWarp<NM, PT>) * (NT / 32);
  auto kern = k_leg_adj_ck<NM, NT, PT>;
  CMBWS_TRY(ensure_dyn_smem((const void*)kern, sm));
  ProfScope ps(PROF_LEG_ADJ, s, 0, leg_work(g, NM));
  kern<<<grd, NT, sm, s>>>(eo, g.A32.as<float>(), g.ls.as<int>(), g.st32.as<float2>(),
                           g.y32.as<float>(), g.ck32.as<float2>(), g.ck_base.as<int64_t>(),
                           g.wt32.as<int2>(), g.nwt32, g.ls_tmin.as<int>(), g.c64.as<double>(),
                           (double2*)out, nlm, L, g.npair);
  CMBWS_LAUNCH_CHECK();
  return CMBWS_OK;
}

int synth_dispatch(const Grid& g, int nmaps, const void* alm, void* F, cudaStream_t s) {
  const int64_t as = nlm_of(g.lmax), fs = (int64_t)g.nring * (g.lmax + 1);
  for (int k0 = 0; k0 < nmaps; k0 += 4) {
    const int nm = nmaps - k0 < 4 ? nmaps - k0 : 4;
    const void* a = (const float2*)alm + k0 * as;
    void* f = (float2*)F + k0 * fs;
    int st = CMBWS_OK;
    switch (nm) {
      case 1: st = launch_synth<1>(g, a, as, f, fs, s); break;
      case 2: st = launch_synth<2>(g, a, as, f, fs, s); break;
      case 3: st = launch_synth<3>(g, a, as, f, fs, s); break;
      default: st = launch_synth<4>(g, a, as, f, fs, s); break;
    }
    if (st != CMBWS_OK) return st;
  }
  return CMBWS_OK;
}

// FP32 adjoints from the adjoint input (eo layout, chunks of 4 maps) that the ring FFT wrote
int adj_dispatch_ck(const Grid& g, int nmaps, const float* eo, double* out, cudaStream_t s) {
  const int64_t nlm = nlm_of(g.lmax), cs = (int64_t)(g.lmax + 1) * g.npair * 4;
  for (int k0 = 0; k0 < nmaps; k0 += 4) {
    const int nm = nmaps - k0 < 4 ? nmaps - k0 : 4;
    const float* e = eo + k0 * cs;
    double* o = out + 2 * k0 * nlm;
    int st = CMBWS_OK;
    switch (nm) {
      case 1: st = launch_adj_ck<1>(g, e, o, s); break;
      case 2: st = launch_adj_ck<2>(g, e, o, s); break;
      case 3: st = launch_adj_ck<3>(g, e, o, s); break;
      default: st = launch_adj_ck<4>(g, e, o, s); break;
    }
    if (st != CMBWS_OK) return st;
  }
  return CMBWS_OK;
}

}  // namespace

int legendre_synth(const Grid& g, int prec, int nmaps, const void* alm, void* F, cudaStream_t s) {
  if (prec == CMBWS_FP64) return legendre_synth_fx(g, nmaps, alm, F, s);
  if (prec == CMBWS_FP32X2) return legendre_synth_df(g, nmaps, alm, F, s);
  if (is_tc(prec)) return legendre_synth_tc(g, prec, nmaps, alm, F, s);
  return synth_dispatch(g, nmaps, alm, F, s);
}

size_t legendre_adjoint_part_bytes(const Grid& g, int prec, int nmaps) {
  // the adjoint input (eo layout) of every map: (L+1) npair 4 scalars per map; the fixed-point
  // stage (FP64) adds one exponent per (map, m)
  const size_t eo = (size_t)nmaps * (g.lmax + 1) * g.npair * 4;
  if (is_f32(prec)) return eo * sizeof(float);
  return eo * 8 + (prec == CMBWS_FP64 ? (size_t)nmaps * (g.lmax + 1) * sizeof(int) : 0);
}

int legendre_adjoint(const Grid& g, int prec, int nmaps, void* part, size_t part_bytes, double* out,
                     cudaStream_t s) {
  if (part_bytes < legendre_adjoint_part_bytes(g, prec, nmaps)) {
    set_error("legendre_adjoint: workspace too small");
    return CMBWS_ERR_ARG;
  }
  if (prec == CMBWS_FP64) {
    int* ee = (int*)((char*)part + (size_t)nmaps * (g.lmax + 1) * g.npair * 4 * 8);
    return legendre_adjoint_fx(g, nmaps, part, ee, out, s);
  }
  if (prec == CMBWS_FP32X2) {
    const int64_t nlm = nlm_of(g.lmax), cs = (int64_t)(g.lmax + 1) * g.npair * 4;
    // at most 3 maps per launch: 4 maps' double-float accumulators exceed the register file
    for (int k0 = 0; k0 < nmaps; k0 += 3) {
      const int nm = nmaps - k0 < 3 ? nmaps - k0 : 3;
      CMBWS_TRY(legendre_adj_df_ck(g, nm, (const float2*)part + k0 * cs, out + 2 * k0 * nlm, s));
    }
    return CMBWS_OK;
  }
  if (prec == CMBWS_BF16 || prec == CMBWS_BF16X3)
    return legendre_adjoint_tc(g, prec, nmaps, (const float*)part, out, s);
  return adj_dispatch_ck(g, nmaps, (const float*)part, out, s);
}

}  // namespace cmbws
