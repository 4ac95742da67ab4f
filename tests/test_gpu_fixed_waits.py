"""The bounded waits of the CMBWS_FP64 kernels: a wait that runs out is reported, without a fault."""
import numpy as np
import pytest

import paper_1710_00621_gb300 as cw
from oracle import grids as og, model as omodel, sht as osht
from tests._gpu import gpu_model, rel_err, to_dev, to_host
from tests._models import oracle_model, tiny_workload

pytestmark = pytest.mark.gpu


# 2 and 7 maps: three and two CTAs per SM
@pytest.mark.parametrize("maps", [2, 7])
@pytest.mark.parametrize("op", ["synth", "analysis"])
def test_wait_runs_out_and_reports_a_timeout(op, maps):
    """Every CTA gives up after 1e5 SM clocks on an mbarrier phase that nothing completes, issues no
    MMA, frees its tensor memory and writes NaN; cmbws_device_status reports CMBWS_ERR_TIMEOUT once,
    and the next call is correct."""
    nside, lmax = 8, 23
    g, o = cw.cmbws_plan_grid(cw.CMBWS_GRID_HEALPIX, nside, lmax), og.healpix(nside)
    rng = np.random.default_rng(maps)
    if op == "synth":
        src, n = rng.standard_normal((maps, (lmax + 1) ** 2)), g.npix
        call = lambda out: cw.cmbws_sht_synth(g, cw.CMBWS_FP64, to_dev(src), out, maps)
        want = [osht.synthesis(o, lmax, a) for a in src]
    else:
        src, n = rng.standard_normal((maps, g.npix)), (lmax + 1) ** 2
        call = lambda out: cw.cmbws_sht_analysis(g, cw.CMBWS_FP64, to_dev(src), out, maps, 1)
        want = [osht.adjoint(o, lmax, f, weighted=True) for f in src]
    out = to_dev(np.zeros((maps, n)))
    cw.cmbws_device_status()                         # clear any earlier record
    cw.cmbws_testing_stall_waits(100000)
    try:
        call(out)
        with pytest.raises(cw.CmbwsError) as e:
            cw.cmbws_device_status()
        assert e.value.code == -7
    finally:
        cw.cmbws_testing_stall_waits(0)
    assert np.isnan(to_host(out)).all()
    cw.cmbws_device_status()                         # the record was cleared
    call(out)
    cw.cmbws_device_status()
    for got, w in zip(to_host(out), want):
        assert rel_err(got, w) < 40 * (lmax + 1) * 2.0 ** -53


def test_solver_reports_a_timed_out_wait_as_timeout():
    work = tiny_workload(15)
    m, inp = oracle_model(work)
    g, _ = gpu_model(work, inp, cw.CMBWS_FP64)
    b = to_dev(omodel.apply_A(m, inp["x_true"]))
    x = to_dev(np.zeros(m.nvec()))
    cw.cmbws_device_status()
    cw.cmbws_testing_stall_waits(100000)
    try:
        rep = cw.cmbws_cg_solve(g, b, x, tol=1e-8, maxiter=50, check=False)
    finally:
        cw.cmbws_testing_stall_waits(0)
    assert rep["code"] == -7, rep
    rep = cw.cmbws_cg_solve(g, b, x, tol=1e-8, maxiter=200)
    assert rep["rel_res"] <= 1e-8
