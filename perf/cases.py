"""The work that a program built on this package gives it, at the sizes it is used at.

Listed cases, smallest to largest, and what each stands for:

* tiny_synth_fp64: the smallest call, one map of the two-component test problem's grid, where
  launches and latency count;
* tiny_solve_fp64: a whole Wiener solve of that problem (GL L = 63, 3 bands, 2 components, 1e-8);
* small_analysis_fp64: weighted analysis of several maps at an odd band-limit on a small HEALPix
  grid, as the coarse levels of the multigrid preconditioner do;
* masked_apply_fp64: y = A x of one masked problem of the batched workload (variable mixing maps
  on a HEALPix grid, bands on Gauss-Legendre grids of odd ring length);
* diff_apply_fp64: y = A x of the differentiable workload (5 GL bands at L = 511, 3 components);
* diff_rhs_fp32: the right-hand side of that problem for a mixed-precision model (its transforms
  are the FP64-accurate double-float ones) with the draws of a constrained realization;
* adjoint_gl1000_fp64: unweighted adjoint of one map at a large odd GL size (the backward pass of
  a differentiable synthesis);
* synth_nside512_fp32x2: double-float synthesis of three bands, as the residual certification does;
* precond_bf16: z = M_PI r of the multi-resolution sky with tensor-core transforms, as inside the
  mixed-precision solver;
* solve_mixed: the benchmark's solve at half its resolution (FP32 A, BF16 M_PI, double-float
  certification);
* adjoint_nside1024_fp32: single-precision adjoint of three full-size bands (one half of A);
* synth_nside1024_fp64: the largest transform, three bands at Nside 1024, L = 3071.

Drawn cases take other sizes, map counts, precisions and models of the same ranges.
"""
import math

import numpy as np
import torch

import paper_1710_00621_gb300 as cw

PRECS = {"fp64": cw.CMBWS_FP64, "fp32x2": cw.CMBWS_FP32X2, "fp32": cw.CMBWS_FP32,
         "tf32": cw.CMBWS_TF32, "bf16": cw.CMBWS_BF16, "bf16x3": cw.CMBWS_BF16X3}
FREQS9 = (30.0, 44.0, 70.0, 100.0, 143.0, 217.0, 353.0, 545.0, 857.0)
ARCMIN = math.pi / (180.0 * 60.0)


def listed():
    return [
        {"name": "tiny_synth_fp64", "op": "synth", "grid": "gl", "n": 64, "lmax": 63, "maps": 1,
         "prec": "fp64"},
        {"name": "tiny_solve_fp64", "op": "solve", "model": "tiny", "size": 63, "prec": "fp64"},
        {"name": "small_analysis_fp64", "op": "analysis", "grid": "healpix", "n": 64, "lmax": 131,
         "maps": 5, "prec": "fp64"},
        {"name": "masked_apply_fp64", "op": "apply", "model": "masked", "size": 297, "prec": "fp64"},
        {"name": "diff_apply_fp64", "op": "apply", "model": "diff", "size": 511, "prec": "fp64"},
        {"name": "diff_rhs_fp32", "op": "rhs", "model": "diff", "size": 511, "prec": "fp32"},
        {"name": "adjoint_gl1000_fp64", "op": "adjoint", "grid": "gl", "n": 1001, "lmax": 1000,
         "maps": 1, "prec": "fp64"},
        {"name": "synth_nside512_fp32x2", "op": "synth", "grid": "healpix", "n": 512, "lmax": 1535,
         "maps": 3, "prec": "fp32x2"},
        {"name": "precond_bf16", "op": "precond", "model": "multires", "size": 512, "prec": "bf16"},
        {"name": "solve_mixed", "op": "solve", "model": "multires", "size": 512, "prec": "fp32"},
        {"name": "adjoint_nside1024_fp32", "op": "adjoint", "grid": "healpix", "n": 1024,
         "lmax": 3071, "maps": 3, "prec": "fp32"},
        {"name": "synth_nside1024_fp64", "op": "synth", "grid": "healpix", "n": 1024, "lmax": 3071,
         "maps": 3, "prec": "fp64"},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(("synth", "synth", "analysis", "adjoint", "adjoint", "apply", "rhs", "precond"))
    prec = rng.choice(("fp64", "fp64", "fp32x2", "fp32x2", "fp32", "tf32", "bf16", "bf16x3"))
    if op in ("synth", "analysis", "adjoint"):
        maps = rng.randint(1, 6)
        if rng.random() < 0.5:
            lmax = _log_int(rng, 31, 1200)
            return {"op": op, "grid": "gl", "n": lmax + 1 + rng.randint(0, 3), "lmax": lmax,
                    "maps": maps, "prec": prec}
        n = _log_int(rng, 16, 700)
        return {"op": op, "grid": "healpix", "n": n, "lmax": rng.randint(2 * n, 3 * n - 1),
                "maps": maps, "prec": prec}
    model = rng.choice(("tiny", "diff", "multires", "masked"))
    size = {"tiny": lambda: _log_int(rng, 31, 200), "diff": lambda: _log_int(rng, 63, 600),
            "multires": lambda: 4 * _log_int(rng, 16, 128),
            "masked": lambda: _log_int(rng, 128, 500)}[model]()
    return {"op": op, "model": model, "size": size, "prec": prec}


# ---- the models ----

def _model(kind, size):
    """(bands, components, masked) of a workload: band = (GHz, grid, n, lmax, FWHM arcmin, sigma,
    contrast of sigma over the sky), component = (lmax, spectral slope of C_l, beta or None,
    reference GHz, crossover)."""
    cmb = (None, None, 1.0, 0.40)
    if kind == "tiny":
        bands = [(f, "gl", size + 1, size, w * 63.0 / size, 10.0, 1.0)
                 for f, w in ((30.0, 60.0), (100.0, 40.0), (353.0, 30.0))]
        return bands, [(size, *cmb), (size, 2.4, 1.6, 353.0, 0.75)], False
    if kind == "diff":
        bands = [(f, "gl", size + 1, size, w * 511.0 / size, 10.0, 3.0) for f, w in
                 ((30.0, 40.0), (70.0, 30.0), (143.0, 20.0), (353.0, 15.0), (857.0, 10.0))]
        return bands, [(size, *cmb), (size, 2.7, -3.0, 30.0, 0.35),
                       (size, 2.4, 1.6, 353.0, 0.75)], False
    if kind == "multires":
        bands = []
        for i, f in enumerate(FREQS9):
            ns = size // (4, 2, 1)[i // 3]
            bands.append((f, "healpix", ns, 3 * ns - 1,
                          33.0 * (5.0 / 33.0) ** (i / 8.0) * 1024.0 / size, 1.0, 3.0))
        return bands, [(2000 * size // 1024, *cmb), (500 * size // 1024, 2.7, -3.0, 30.0, 0.35),
                       (3000 * size // 1024, 2.4, 1.6, 353.0, 0.75)], False
    fw = math.sqrt(8.0 * math.log(2.0)) / ARCMIN
    bands = [(f, "gl", size + 1, size, c / size * fw, 10.0, 1.0)
             for f, c in ((30.0, 2.0), (100.0, 1.6), (353.0, 1.3))]
    return bands, [(size, *cmb), (size, 2.4, 1.6, 353.0, 0.75)], True


def _mix_nside(lmax):
    ns = 1
    while 3 * ns - 1 < lmax:
        ns *= 2
    return ns


def _beam(fwhm, lmax):
    s = fwhm * ARCMIN / math.sqrt(8.0 * math.log(2.0))
    l = np.arange(lmax + 1, dtype=np.float64)
    return np.exp(-0.5 * l * (l + 1.0) * s * s)


def _cl_shape(slope, lmax):
    l = np.maximum(np.arange(lmax + 1, dtype=np.float64), 1.0 if slope else 2.0)
    return l ** -slope if slope else 1.0 / (l * (l + 1.0))


def _q(bands, comps):
    return np.array([[1.0 if c[2] is None else (b[0] / c[3]) ** c[2] for c in comps]
                     for b in bands])


class _Ring:
    """Ring geometry of a grid, from its definition (the same pixels as the package's grids)."""

    def __init__(self, kind, n, lmax):
        if kind == "gl":
            x, w = np.polynomial.legendre.leggauss(n)
            self.z, nphi = x[::-1].copy(), 2 * lmax + 1
            self.nphi = np.full(n, nphi)
            self.phi0 = np.zeros(n)
            self.w = w[::-1] * 2.0 * np.pi / nphi
        else:
            i = np.arange(1, 4 * n)
            ip = np.minimum(i, 4 * n - i)
            cap = ip < n
            z = np.where(cap, 1.0 - ip * ip / (3.0 * n * n), 4.0 / 3.0 - 2.0 * ip / (3.0 * n))
            self.z = np.where(i > 2 * n, -z, z)
            self.nphi = np.where(cap, 4 * ip, 4 * n)
            self.phi0 = np.where(cap, np.pi / self.nphi, np.where((ip - n) % 2 == 0,
                                                                 np.pi / (4.0 * n), 0.0))
            self.w = np.full(i.size, 4.0 * np.pi / (12.0 * n * n))
        self.off = np.concatenate([[0], np.cumsum(self.nphi)])
        self.npix, self.nring = int(self.off[-1]), self.z.size

    def pixels(self):
        """(x, y, z) of every pixel, and each pixel's ring, on the GPU."""
        d = "cuda"
        ring = torch.repeat_interleave(torch.arange(self.nring, device=d),
                                       torch.as_tensor(self.nphi, device=d))
        k = torch.arange(self.npix, device=d) - torch.as_tensor(self.off[:-1], device=d)[ring]
        ph = (torch.as_tensor(self.phi0, device=d)[ring]
              + 2.0 * math.pi * k / torch.as_tensor(self.nphi, device=d)[ring])
        z = torch.as_tensor(self.z, device=d)[ring]
        s = torch.sqrt((1.0 - z * z).clamp_min(0.0))
        return s * torch.cos(ph), s * torch.sin(ph), z


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(1710_00621 + seed)


def _normal(n, gen):
    return torch.randn(n, dtype=torch.float64, device="cuda", generator=gen)


def _ell(lmax):
    """l of every packed coefficient: the m = 0 block, then the cos and sin blocks of each m."""
    l = torch.arange(lmax + 1, device="cuda")
    ms = torch.cat([l[:1], l[1:].repeat_interleave(2)])
    lens = lmax + 1 - ms
    start = torch.cumsum(lens, 0) - lens
    return torch.arange((lmax + 1) ** 2, device="cuda") - torch.repeat_interleave(start - ms, lens)


def _sky(lmax, slope, gen, maps=1):
    """Gaussian coefficients of the spectrum l^-slope (None: 1 / l(l+1))."""
    s = torch.as_tensor(np.sqrt(_cl_shape(slope, lmax)), device="cuda")
    return _normal(maps * (lmax + 1) ** 2, gen) * s[_ell(lmax)].repeat(maps)


def _depth(ring, sigma, contrast, gen):
    """Noise rms per pixel: sigma times contrast^s, s a smooth pattern in [0, 1]."""
    if contrast == 1.0:
        return torch.full((ring.npix,), sigma, dtype=torch.float64, device="cuda")
    x, y, z = ring.pixels()
    c = _normal(9, gen).tolist()
    s = (c[0] * x + c[1] * y + c[2] * z + c[3] * x * y + c[4] * y * z + c[5] * x * z
         + c[6] * x * x * z + c[7] * y * y * x + c[8] * z ** 4)
    lo, hi = s.min(), s.max()
    return sigma * contrast ** ((s - lo) / (hi - lo))


def _model_inputs(case, seed):
    """Every input of a model case: maps on the GPU, spectra and mixing as numpy."""
    gen = _gen(seed)
    bands, comps, masked = _model(case["model"], case["size"])
    rings = {}
    for b in bands:
        rings.setdefault(b[1:4], _Ring(*b[1:4]))
    rb = [rings[b[1:4]] for b in bands]
    sig = [_depth(r, b[5], b[6], gen) for r, b in zip(rb, bands)]
    tau = [1.0 / (s * s) for s in sig]
    beams, q = [_beam(b[4], b[3]) for b in bands], _q(bands, comps)
    # prior amplitudes: 1 / C_l meets the data term at l = crossover L_k
    level = [float((t.sum() / sum(r.w * r.nphi))) for t, r in zip(tau, rb)]
    cls = []
    for k, (lk, slope, _, _, cross) in enumerate(comps):
        lx = max(2, round(cross * lk))
        d = sum(q[i, k] ** 2 * beams[i][lx] ** 2 * level[i] for i, b in enumerate(bands)
                if lx <= b[3])
        shape = _cl_shape(slope, lk)
        cls.append(shape / (d * shape[lx]))
    inp = {"bands": bands, "comps": comps, "rings": rb, "tau": tau, "beams": beams, "q": q,
           "cls": cls, "mix": None, "gen": gen, "sig": sig}
    if masked:
        # a galactic-band mask carried by the mixing maps
        ns = _mix_nside(case["size"])
        inp["mix_ring"], inp["mix_n"] = _Ring("healpix", ns, case["size"]), ns
        z = inp["mix_ring"].pixels()[2]
        b0 = 0.05 + 0.25 * float(torch.rand(1, device="cuda", generator=gen))
        m = (z.abs() >= b0).to(torch.float64)
        inp["mix"] = [[float(q[i, k]) * m for k in range(len(comps))] for i in range(len(bands))]
    inp["x"] = torch.cat([_normal((c[0] + 1) ** 2, gen)
                          * torch.as_tensor(np.sqrt(cl), device="cuda")[_ell(c[0])]
                          for c, cl in zip(comps, cls)])
    return inp


def _plan(kind, n, lmax):
    return cw.cmbws_plan_grid(cw.CMBWS_GRID_GL if kind == "gl" else cw.CMBWS_GRID_HEALPIX, n, lmax)


def _prepare_transform(case, seed):
    gen = _gen(seed)
    g = _plan(case["grid"], case["n"], case["lmax"])
    nm, nalm = case["maps"], (case["lmax"] + 1) ** 2
    alm = _sky(case["lmax"], 2.0, gen, nm)
    if case["op"] == "synth":
        src, dst = alm, torch.empty(nm * g.npix, dtype=torch.float64, device="cuda")
    else:
        src, dst = _normal(nm * g.npix, gen), torch.empty_like(alm)
        assert dst.numel() == nm * nalm
    return {"case": case, "grid": g, "src": src, "dst": dst, "prec": PRECS[case["prec"]]}


def _prepare_model(case, seed):
    inp = _model_inputs(case, seed)
    plans = {}
    for b in inp["bands"]:
        if b[1:4] not in plans:
            plans[b[1:4]] = _plan(*b[1:4])
    grids = [plans[b[1:4]] for b in inp["bands"]]
    mg = mm = None
    if inp["mix"]:
        g = _plan("healpix", inp["mix_n"], case["size"])
        mm, mg = inp["mix"], [[g] * len(inp["comps"]) for _ in inp["bands"]]
    m = cw.cmbws_model_create([c[0] for c in inp["comps"]], grids, inp["beams"], inp["cls"],
                              inp["tau"], inp["q"], PRECS[case["prec"]], mix_grids=mg, mix_maps=mm)
    st = {"case": case, "model": m, "x": inp["x"], "out": torch.empty_like(inp["x"])}
    if case["op"] in ("rhs", "solve"):
        st.update(_data(case, inp))
    if case["op"] == "solve":
        st["b"] = torch.empty_like(inp["x"])
        if case["prec"] != "fp64":
            cw.cmbws_model_set_precond_prec(m, cw.CMBWS_BF16)
        st["opts"] = ({"tol": 1e-8, "cert_prec": cw.CMBWS_FP64} if case["prec"] == "fp64" else
                      {"tol": 1e-6, "cert_prec": cw.CMBWS_FP32X2})
    return st


def _data(case, inp):
    """Band maps d (noise on a white signal), and the draws of a constrained realization."""
    gen = inp["gen"]
    d = [s * _normal(s.numel(), gen) * 1.5 for s in inp["sig"]]
    if case["op"] == "solve":
        return {"d": d, "w1": None, "w2": None}
    return {"d": d, "w1": [_normal(s.numel(), gen) for s in inp["sig"]],
            "w2": _normal(inp["x"].numel(), gen)}


def prepare(case, seed):
    return _prepare_model(case, seed) if "model" in case else _prepare_transform(case, seed)


def run(state):
    case, op = state["case"], state["case"]["op"]
    if op == "synth":
        cw.cmbws_sht_synth(state["grid"], state["prec"], state["src"], state["dst"], case["maps"])
        return state["dst"]
    if op in ("analysis", "adjoint"):
        cw.cmbws_sht_analysis(state["grid"], state["prec"], state["src"], state["dst"],
                              case["maps"], weighted=1 if op == "analysis" else 0)
        return state["dst"]
    m = state["model"]
    if op == "apply":
        cw.cmbws_apply_A(m, state["x"], state["out"])
    elif op == "precond":
        cw.cmbws_apply_precond(m, state["x"], state["out"])
    elif op == "rhs":
        cw.cmbws_rhs(m, state["d"], state["out"], state["w1"], state["w2"])
    else:
        # one Wiener filter from the band maps, from a zero initial guess
        cw.cmbws_rhs(m, state["d"], state["b"])
        state["out"].zero_()
        cw.cmbws_cg_solve(m, state["b"], state["out"], **state["opts"])
    return state["out"]


# ---- the work a case cannot do without ----

def _sht_flops(kind, n, lmax, maps):
    """4 flops of recurrence plus 4 per map for every (l, m, ring pair), and the ring FFTs."""
    nring = n if kind == "gl" else 4 * n - 1
    npix = n * (2 * lmax + 1) if kind == "gl" else 12 * n * n
    legendre = 4.0 * (1 + maps) * ((nring + 1) // 2) * (lmax + 1) * (lmax + 2) / 2
    return legendre + maps * 2.5 * npix * math.log2(max(2, npix / nring))


def work(case):
    if "model" not in case:
        r = (case["grid"], case["n"], case["lmax"])
        npix = r[1] * (2 * r[2] + 1) if r[0] == "gl" else 12 * r[1] * r[1]
        return {"bytes": 8.0 * case["maps"] * (npix + (r[2] + 1) ** 2),
                "flops": _sht_flops(*r, case["maps"])}
    bands, comps, masked = _model(case["model"], case["size"])
    nvec = sum((c[0] + 1) ** 2 for c in comps)
    npix = sum(b[2] * (2 * b[3] + 1) if b[1] == "gl" else 12 * b[2] ** 2 for b in bands)
    groups = {}
    for b in bands:
        groups[b[1:4]] = groups.get(b[1:4], 0) + 1
    one = sum(_sht_flops(*g, n) for g, n in groups.items())
    mix = 0.0
    if masked:
        pairs = len(bands) * len(comps)
        mix = _sht_flops("healpix", _mix_nside(case["size"]), case["size"], pairs)
    apply = 2 * one + 4 * mix
    # the solves' iterations (one apply of A and of M_PI each): 16 to 1e-8 and 9 to 1e-6 with
    # two certification applies
    n_it = {"fp64": (16, 1)}.get(case["prec"], (9, 2))
    flops = {"apply": apply, "precond": 2 * one, "rhs": one + 2 * mix,
             "solve": one + n_it[0] * (apply + 2 * one) + n_it[1] * apply}[case["op"]]
    reads = {"apply": 2 * nvec + npix, "precond": 2 * nvec + npix, "rhs": 2 * nvec + 3 * npix,
             "solve": nvec + 2 * npix}[case["op"]]
    if masked:
        reads += len(bands) * len(comps) * 12 * _mix_nside(case["size"]) ** 2
    return {"bytes": 8.0 * reads, "flops": flops}


# ---- the same results in plain 64-bit torch ----

class _Exact:
    """Spherical harmonic transforms of one ring grid in 64 bits: the three-term recurrence of the
    orthonormal Legendre functions over all (m, ring) at once (values carried with an exponent,
    as lambda_mm underflows near the poles), and one FFT per ring."""

    def __init__(self, ring, lmax):
        self.r, self.L = ring, lmax
        self.half = (ring.nring + 1) // 2
        self.z = torch.as_tensor(ring.z[:self.half], device="cuda")
        # 1 - z, which keeps its relative precision near the pole
        self.y = 2.0 * torch.sin(0.5 * torch.arccos(self.z)) ** 2

    def _lambdas(self):
        """Yields (l, m0, lambda[m <= l][ring of the north half])."""
        L, d = self.L, "cuda"
        s = torch.sqrt(self.y * (2.0 - self.y))
        # lambda_mm by its product in floating point with the exponent beside it
        mant, ex = [], []
        v = torch.full_like(self.z, math.sqrt(1.0 / (4.0 * math.pi)))
        k = torch.zeros_like(self.z)
        for mm in range(L + 1):
            if mm:
                v = v * (math.sqrt((2.0 * mm + 1.0) / (2.0 * mm)) * s)
                small = v.abs() < 2.0 ** -300
                v = torch.where(small, v * 2.0 ** 300, v)
                k = k - small.to(v.dtype)
            mant.append(v)
            ex.append(k)
        p1 = torch.stack(mant)   # lambda_{l-1}, scaled by 2^(300 ex)
        ex = torch.stack(ex)
        p0 = torch.zeros_like(p1)
        seed = p1.clone()
        for l in range(L + 1):
            if l:
                mm = torch.arange(l, dtype=torch.float64, device=d)[:, None]
                a = torch.sqrt((4.0 * l * l - 1.0) / (l * l - mm * mm))
                b = torch.sqrt(((l - 1.0) ** 2 - mm * mm) / (4.0 * (l - 1.0) ** 2 - 1.0)) \
                    if l > 1 else torch.zeros_like(mm)
                new = a * ((p1[:l] - self.y * p1[:l]) - b * p0[:l])
                p0[:l] = p1[:l]
                p1[:l] = new
                if l % 4 == 0:
                    big = (new.abs() > 2.0 ** 100) & (ex[:l] < 0)
                    f = torch.exp2(-300.0 * big.to(torch.float64))
                    p0[:l] *= f
                    p1[:l] *= f
                    ex[:l] += big
                p1[l], p0[l] = seed[l], 0.0
            yield l, torch.where(ex[:l + 1] >= 0, p1[:l + 1], torch.zeros_like(p1[:l + 1]))

    def _unpack(self, alm):
        """packed [maps, (L+1)^2] -> (cos, sin) dense [maps, l, m]."""
        L, nm = self.L, alm.shape[0]
        c = torch.zeros(nm, L + 1, L + 1, dtype=torch.float64, device="cuda")
        s = torch.zeros_like(c)
        o = 0
        for m in range(L + 1):
            n = L + 1 - m
            c[:, m:, m] = alm[:, o:o + n]
            o += n
            if m:
                s[:, m:, m] = alm[:, o:o + n]
                o += n
        return c, s

    def _pack(self, c, s):
        out = []
        for m in range(self.L + 1):
            out.append(c[:, m:, m])
            if m:
                out.append(s[:, m:, m])
        return torch.cat(out, 1)

    def synth(self, alm):
        L, h, r = self.L, self.half, self.r
        c, s = self._unpack(alm)
        nm = alm.shape[0]
        # sums over even and odd l - m separately: the south ring has their difference
        F = torch.zeros(2, nm, L + 1, h, dtype=torch.complex128, device="cuda")
        par = torch.arange(L + 1, device="cuda") % 2
        for l, lam in self._lambdas():
            a = torch.complex(c[:, l, :l + 1], s[:, l, :l + 1])[:, :, None]
            odd = (par[:l + 1] != l % 2).to(torch.float64)[:, None]
            F[0, :, :l + 1] += a * (lam * (1.0 - odd))
            F[1, :, :l + 1] += a * (lam * odd)
        maps = torch.empty(nm, r.npix, dtype=torch.float64, device="cuda")
        m = torch.arange(L + 1, device="cuda")
        wm = 1.0 + (math.sqrt(2.0) - 1.0) * (m > 0).to(torch.float64)
        for i in range(r.nring):
            n, p = int(r.nphi[i]), min(i, r.nring - 1 - i)
            f = F[0, :, :, p] + (F[1, :, :, p] if i < h else -F[1, :, :, p])
            # sum_m w_m (C cos m phi + S sin m phi) = Re sum_m w_m (C - i S) e^{i m phi}
            g = f.conj() * (wm * torch.exp(1j * float(r.phi0[i]) * m.to(torch.float64)))
            H = torch.zeros(nm, n, dtype=torch.complex128, device="cuda").index_add_(1, m % n, g)
            maps[:, r.off[i]:r.off[i] + n] = (torch.fft.ifft(H, dim=1) * n).real
        return maps

    def adjoint(self, maps, weighted):
        L, h, r = self.L, self.half, self.r
        nm = maps.shape[0]
        m = torch.arange(L + 1, device="cuda")
        wm = 1.0 + (math.sqrt(2.0) - 1.0) * (m > 0).to(torch.float64)
        G = torch.zeros(2, nm, L + 1, h, dtype=torch.complex128, device="cuda")
        for i in range(r.nring):
            n, p = int(r.nphi[i]), min(i, r.nring - 1 - i)
            f = maps[:, r.off[i]:r.off[i] + n] * (float(r.w[i]) if weighted else 1.0)
            Z = torch.fft.fft(f.to(torch.complex128), dim=1)[:, m % n]
            g = (Z * (wm * torch.exp(-1j * float(r.phi0[i]) * m.to(torch.float64)))).conj()
            G[0, :, :, p] += g
            G[1, :, :, p] += g if i < h else -g
        c = torch.zeros(nm, L + 1, L + 1, dtype=torch.float64, device="cuda")
        s = torch.zeros_like(c)
        par = torch.arange(L + 1, device="cuda") % 2
        for l, lam in self._lambdas():
            odd = (par[:l + 1] != l % 2)[None, :, None]
            v = (torch.where(odd, G[1, :, :l + 1], G[0, :, :l + 1]) * lam).sum(-1)
            c[:, l, :l + 1], s[:, l, :l + 1] = v.real, v.imag
        return self._pack(c, s)


def _resize(a, l_from, l_to):
    """Packed coefficients of another band-limit (zero-padded or cut)."""
    if l_from == l_to:
        return a
    out = torch.zeros((l_to + 1) ** 2, dtype=torch.float64, device="cuda")
    i = j = 0
    for m in range(min(l_from, l_to) + 1):
        for _ in range(1 if m == 0 else 2):
            n = min(l_from, l_to) + 1 - m
            out[j:j + n] = a[i:i + n]
            i += l_from + 1 - m
            j += l_to + 1 - m
    return out


class _ExactModel:
    def __init__(self, case, seed):
        self.i = _model_inputs(case, seed)
        self.data = _data(case, self.i)
        self.sht = {}
        for b, r in zip(self.i["bands"], self.i["rings"]):
            self.sht.setdefault(b[1:4], _Exact(r, b[3]))
        self.lk = [c[0] for c in self.i["comps"]]
        if self.i["mix"]:
            self.msht = _Exact(self.i["mix_ring"], case["size"])
            r = self.i["mix_ring"]
            self.mw = torch.repeat_interleave(torch.as_tensor(r.w, device="cuda"),
                                              torch.as_tensor(r.nphi, device="cuda"))

    def split(self, x):
        return list(torch.split(x, [(l + 1) ** 2 for l in self.lk]))

    def beam(self, nu, a):
        l = self.i["bands"][nu][3]
        return a * torch.as_tensor(self.i["beams"][nu], device="cuda")[_ell(l)]

    def prior(self, x, power):
        return torch.cat([a * torch.as_tensor(cl ** power, device="cuda")[_ell(l)]
                          for a, cl, l in zip(self.split(x), self.i["cls"], self.lk)])

    def mixed(self, jobs):
        """Q~ a for every (nu, k, a): synthesis, the mixing map, weighted analysis."""
        maps = self.msht.synth(torch.stack([a for _, _, a in jobs]))
        for j, (nu, k, _) in enumerate(jobs):
            maps[j] *= self.i["mix"][nu][k]
        return self.msht.adjoint(maps, True)

    def band_fields(self, x):
        xs, out = self.split(x), []
        nb, nc = len(self.i["bands"]), len(self.lk)
        mixed = self.mixed([(nu, k, xs[k]) for nu in range(nb) for k in range(nc)]) \
            if self.i["mix"] else None
        for nu, b in enumerate(self.i["bands"]):
            a = sum((mixed[nu * nc + k] if self.i["mix"] else
                     float(self.i["q"][nu, k]) * _resize(xs[k], self.lk[k], b[3]))
                    for k in range(nc))
            out.append(self.beam(nu, a))
        return out

    def gather(self, u):
        """sum_nu Q~^T B u_nu"""
        nb, nc = len(self.i["bands"]), len(self.lk)
        bu = [self.beam(nu, a) for nu, a in enumerate(u)]
        if self.i["mix"]:
            t = self.mixed([(nu, k, bu[nu]) for nu in range(nb) for k in range(nc)])
            return torch.cat([sum(t[nu * nc + k] for nu in range(nb)) for k in range(nc)])
        return torch.cat([sum(float(self.i["q"][nu, k])
                              * _resize(bu[nu], self.i["bands"][nu][3], self.lk[k])
                              for nu in range(nb)) for k in range(nc)])

    def chain(self, fields, factors, back_only=False):
        """Y^T (factor * Y a) per band, the bands of one grid together."""
        out = [None] * len(fields)
        for key, sht in self.sht.items():
            nus = [nu for nu, b in enumerate(self.i["bands"]) if b[1:4] == key]
            maps = (torch.stack([fields[nu] for nu in nus]) if back_only else
                    sht.synth(torch.stack([fields[nu] for nu in nus])))
            res = sht.adjoint(maps * torch.stack([factors[nu] for nu in nus]), False)
            for j, nu in enumerate(nus):
                out[nu] = res[j]
        return out

    def apply(self, x):
        return self.prior(x, -1.0) + self.gather(self.chain(self.band_fields(x), self.i["tau"]))

    def rhs(self):
        d, w1, w2 = self.data["d"], self.data["w1"], self.data["w2"]
        t = self.i["tau"]
        pix = [a * b if w1 is None else a * b + w * torch.sqrt(b)
               for a, b, w in zip(d, t, w1 or d)]
        b = self.gather(self.chain(pix, [torch.ones_like(p) for p in pix], back_only=True))
        return b if w2 is None else b + self.prior(w2, -0.5)

    def precond(self, r):
        bands, nc = self.i["bands"], len(self.lk)
        nb, q = len(bands), self.i["q"].copy()
        if self.i["mix"]:
            q = np.array([[float((v * v).sum() / v.sum()) for v in row] for row in self.i["mix"]])
        pw = [torch.repeat_interleave(torch.as_tensor(g.w, device="cuda"),
                                      torch.as_tensor(g.nphi, device="cuda"))
              for g in self.i["rings"]]
        alpha = [math.sqrt(float((t / w).square().sum() / (t / w).sum()))
                 for t, w in zip(self.i["tau"], pw)]
        lc = max(self.lk)
        up = np.zeros((lc + 1, nc, nb + nc))
        for l in range(lc + 1):
            act = [k for k in range(nc) if l <= self.lk[k]]
            u = np.zeros((nb + nc, len(act)))
            for j, k in enumerate(act):
                for nu in range(nb):
                    if l <= bands[nu][3]:
                        u[nu, j] = alpha[nu] * self.i["beams"][nu][l] * q[nu, k]
                u[nb + k, j] = self.i["cls"][k][l] ** -0.5
            up[l, act] = np.linalg.pinv(u, rcond=1e-12)
        up = torch.as_tensor(up, device="cuda")
        rs = self.split(r)

        def per_l(a, l_from, l_to, c, j):
            top = max(lc, l_to)
            f = torch.zeros(top + 1, dtype=torch.float64, device="cuda")
            f[:lc + 1] = up[:, c, j]
            return _resize(a, l_from, l_to) * f[_ell(l_to)]

        rows = [sum(per_l(rs[c], self.lk[c], bands[nu][3], c, nu) for c in range(nc))
                for nu in range(nb)]
        fac = [alpha[nu] ** 2 * pw[nu] ** 2 / self.i["tau"][nu] for nu in range(nb)]
        t = self.chain(rows, fac)
        pr = [sum(per_l(rs[c], self.lk[c], self.lk[k], c, nb + k) for c in range(nc))
              for k in range(nc)]
        return torch.cat([sum(per_l(t[nu], bands[nu][3], self.lk[c], c, nu) for nu in range(nb))
                          + sum(per_l(pr[k], self.lk[k], self.lk[c], c, nb + k)
                                for k in range(nc)) for c in range(nc)])

    def solve(self):
        """Cholesky solution of the dense system (small band-limits, one grid per problem)."""
        nc, L = len(self.lk), self.lk[0]
        n = (L + 1) ** 2
        A = torch.diag(self.prior(torch.ones(nc * n, dtype=torch.float64, device="cuda"), -1.0))
        for nu, b in enumerate(self.i["bands"]):
            sht = self.sht[b[1:4]]
            Y = torch.cat([sht.synth(e) for e in
                           torch.eye(n, dtype=torch.float64, device="cuda").split(512)])
            Y *= torch.as_tensor(self.i["beams"][nu], device="cuda")[_ell(L)][:, None]
            G = (Y * self.i["tau"][nu]) @ Y.T
            A += torch.kron(torch.as_tensor(np.outer(self.i["q"][nu], self.i["q"][nu]),
                                            device="cuda"), G)
        return torch.cholesky_solve(self.rhs()[:, None], torch.linalg.cholesky(A))[:, 0]


def exact(case, seed):
    if "model" not in case:
        gen = _gen(seed)
        ring = _Ring(case["grid"], case["n"], case["lmax"])
        sht, nm = _Exact(ring, case["lmax"]), case["maps"]
        alm = _sky(case["lmax"], 2.0, gen, nm)
        if case["op"] == "synth":
            return sht.synth(alm.reshape(nm, -1)).reshape(-1)
        return sht.adjoint(_normal(nm * ring.npix, gen).reshape(nm, -1),
                           case["op"] == "analysis").reshape(-1)
    if case["op"] == "solve" and (case["model"] != "tiny" or case["size"] > 80):
        return None
    m = _ExactModel(case, seed)
    return {"apply": lambda: m.apply(m.i["x"]), "precond": lambda: m.precond(m.i["x"]),
            "rhs": m.rhs, "solve": m.solve}[case["op"]]()
