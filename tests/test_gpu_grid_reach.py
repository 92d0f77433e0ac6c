"""Rows out of reach of a source grid, with weights so large that what is left
out could be seen: a kernel value below 2^-126 is not held in FP32, and the grid
kernels leave such pairs out (scaled squared distance t above 127), so a row's sum
and a source's gradient may lack 2^-126 of the sum of absolute weights, on top of
the matvec tolerance (2e-5 of the sum of absolute terms, and four FP32 roundings of
an exponent of up to 150). Rows at t = 100 are in reach, at 130 and 150 not."""
import numpy as np
import pytest

from paper_2105_09465_gb300 import api, workloads as W
from tests.gpu_util import MATVEC_REL, assert_close_tol, dev, host, need_gpu

pytestmark = pytest.mark.gpu

REL = MATVEC_REL + 4 * 150 * 2.0**-24


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    need_gpu()


@pytest.mark.parametrize("ell", [0.05, 0.4])
@pytest.mark.parametrize("big", [1.0, 1e30])
def test_rows_beyond_the_reach(orc, ell, big):
    rng = np.random.default_rng(5)
    yg = W.Grid(40, 30, 1, 0.05)
    y = orc.grid_points(*yg.astuple())
    edge, unit = y[:, 0].max(), ell * np.sqrt(2.0 / np.log2(np.e))  # t = (d / unit)^2
    far = [(edge + unit * np.sqrt(t), 0.025) for t in (100.0, 130.0, 150.0)]
    x = np.concatenate([rng.uniform(-0.7, 0.7, (300, 2)), far]).astype(np.float32)
    v = (big * rng.standard_normal(yg.n)).astype(np.float32)
    q, s = api.Points(xy=dev(x)), api.Points(grid=yg)
    want, ab = orc.kernel_matvec(x, y, v, ell, 1.0)
    tol = REL * ab + 2.0**-126 * np.abs(v.astype(np.float64)).sum()
    out, mom = api.gp_kernel_matvec_train(q, s, dev(v), ell, 1.0)
    for got in (api.gp_kernel_matvec(q, s, dev(v), ell, 1.0), out):
        assert_close_tol(host(got), want, tol, what="rows")
    # the column sums: d_v_j = sum_i k_ij g_i, g large at the far rows
    g = rng.standard_normal(len(x)).astype(np.float32)
    g[300:] *= np.float32(big)
    dv = api.gp_kernel_matvec_bwd(q, s, dev(v), ell, 1.0, dev(g), want=("v",), moments=mom)["v"]
    want, ab = orc.kernel_matvec(y, x, g, ell, 1.0)
    assert_close_tol(host(dv), want, REL * ab + 2.0**-126 * np.abs(g.astype(np.float64)).sum(), what="columns")
