"""The dot products of the solver at the sizes where their grid changes."""
import math

import numpy as np
import pytest

import paper_1710_00621_gb300 as cw
from tests._gpu import gpu_model, to_dev, to_host
from tests._models import oracle_model, tiny_workload

pytestmark = pytest.mark.gpu


def _norm(v):
    return math.sqrt(math.fsum(v * v))


@pytest.mark.parametrize("L", [10, 11, 361, 362])
def test_sums_at_the_edges_of_the_reduction_grid(L):
    """2 (L+1)^2 unknowns around one block (256) and the largest grid (1024 blocks).  The sums of
    squares are trees of short chains: within 30 roundings of the exact ones."""
    work = tiny_workload(L)
    m, inp = oracle_model(work)
    g, _ = gpu_model(work, inp)
    n = m.nvec()
    rng = np.random.default_rng(L)
    b, t = rng.standard_normal(n), rng.standard_normal(n)
    cw.cmbws_cg_track_error(g, to_dev(t))
    x = to_dev(np.zeros(n))
    rep = cw.cmbws_cg_solve(g, to_dev(b), x, tol=1e-14, maxiter=1, check=False)
    assert rep["iters"] == 1
    ax = to_dev(np.zeros(n))
    cw.cmbws_apply_A(g, x, ax)
    _, err = cw.cmbws_cg_history(g)
    tol = 30 * 2.0 ** -53
    ref = _norm(b - to_host(ax)) / _norm(b)
    assert abs(rep["rel_res"] - ref) <= tol * ref
    ref = _norm(to_host(x) - t) / _norm(t)
    assert abs(err[0] - ref) <= tol * ref
