"""The ray-trace backward's subhalo sums where each tile picks its own phase
count and takes the local expansion at any subhalo count: counts on both sides
of a group of 128 slots, tiles of few and of many points, grids and explicit
points. Against the FP64 oracle within 2e-5 of the sum of absolute terms (the
repository's gradient tolerance), and repeated calls bit for bit."""
import numpy as np
import pytest
import torch

from paper_2105_09465_gb300 import api, workloads as W
from tests.gpu_util import GRAD_REL, assert_close_tol, dev, host, need_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    need_gpu()


@pytest.mark.parametrize("n_sub", [1, 2, 17, 63, 65, 127, 129, 200, 257])
@pytest.mark.parametrize("side,explicit", [(7, False), (23, True), (60, False), (60, True)])
def test_phases_and_expansion(orc, n_sub, side, explicit):
    rng = np.random.default_rng(100 * side + n_sub)
    g = W.Grid(side, side + 3, 2, 0.12)
    lens = W.draw_lens(rng)
    sub = W.draw_subhalos(rng, n_sub, lens, 1e7, 1e10)
    xi = orc.grid_points(*g.astuple())
    d = rng.standard_normal((g.n, 2)).astype(np.float32)
    q = api.Points(xy=dev(xi), lens=lens, sub=dev(sub)) if explicit else api.Points(grid=g, lens=lens, sub=dev(sub))
    dl, ds = api.lens_raytrace_vjp(q, dev(d))
    dl2, ds2 = api.lens_raytrace_vjp(q, dev(d))
    assert torch.equal(dl, dl2) and torch.equal(ds, ds2)
    rl, rs, al, asub = orc.raytrace_vjp(xi.astype(np.float64), lens.astuple(), sub, d.astype(np.float64), with_abs=True)
    assert_close_tol(host(dl), rl, GRAD_REL * al, what="lens")
    assert_close_tol(host(ds), rs, GRAD_REL * asub, what="subhalos")
