"""When the tables of the CMBWS_FP64 Legendre stage are built, and what they hold until then."""
import numpy as np
import pytest

import paper_1710_00621_gb300 as cw
from oracle import model as omodel
from tests._gpu import gpu_model, rel_err, to_dev, to_host
from tests._models import oracle_model, tiny_workload

pytestmark = pytest.mark.gpu


def _free():
    import torch
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


def test_plan_holds_one_checkpoint_table():
    """A grid planned for FP32 transforms holds the FP32 checkpoints (8 bytes per 8 values of l of every
    pair), 28 bytes of starts per (m, pair), 32 of recurrence tables per (l, m), FFT tables in three
    arithmetics (40 bytes per entry: chirps, phases and filters of each ring length) and less than 64 MB
    of the rest; its first FP64 transform adds as many bytes of checkpoints again."""
    n, lmax = 512, 1535
    to_dev(np.zeros(1))
    before = _free()
    g = cw.cmbws_plan_grid(cw.CMBWS_GRID_HEALPIX, n, lmax)
    planned = _free()
    npair = 2 * n
    ck = 8 * npair * sum((lmax - m + 8) // 8 for m in range(lmax + 1))
    nlm = (lmax + 1) * (lmax + 2) // 2
    fft = 40 * sum(2 * int(k) + (1 << (2 * int(k) - 2).bit_length()) for k in set(g.nphi))
    assert before - planned < ck + 28 * (lmax + 1) * npair + 32 * nlm + fft + (64 << 20)
    alm = to_dev(np.zeros((lmax + 1) ** 2))
    out = to_dev(np.zeros(g.npix))
    cw.cmbws_sht_synth(g, cw.CMBWS_FP32, alm, out, 1)
    used = _free()
    cw.cmbws_sht_synth(g, cw.CMBWS_FP64, alm, out, 1)
    assert used - _free() > 0.9 * ck


def test_first_apply_of_an_fp64_model_can_be_captured():
    import torch
    w = tiny_workload(31)
    m, inp = oracle_model(w)
    gm, _ = gpu_model(w, inp, cw.CMBWS_FP64)
    x = to_dev(inp["x_true"])
    y = torch.zeros_like(x)
    s = torch.cuda.Stream()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=s):
        cw.cmbws_apply_A(gm, x, y, stream=s.cuda_stream)
    graph.replay()
    assert rel_err(to_host(y), omodel.apply_A(m, inp["x_true"])) < 1e-12


def test_first_fp64_transform_can_be_captured():
    """The tables are then built beside the capture."""
    import torch
    n, lmax = 400, 1199  # 0.6 GB of tables: not built with the plan
    alm = to_dev(np.random.default_rng(1).standard_normal((2, (lmax + 1) ** 2)))
    out = to_dev(np.zeros((2, 12 * n * n)))
    grids = [cw.cmbws_plan_grid(cw.CMBWS_GRID_HEALPIX, n, lmax) for _ in range(2)]
    cw.cmbws_sht_synth(grids[0], cw.CMBWS_FP64, alm, out, 1)
    eager = to_host(out)[0].copy()
    cw.cmbws_sht_synth(grids[1], cw.CMBWS_FP32, alm, out, 2)  # workspaces as large as one FP64 map's
    assert rel_err(to_host(out)[0], eager) < 1e-3
    s = torch.cuda.Stream()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=s):
        cw.cmbws_sht_synth(grids[1], cw.CMBWS_FP64, alm, out, 1, stream=s.cuda_stream)
    graph.replay()
    assert np.array_equal(to_host(out)[0], eager)
