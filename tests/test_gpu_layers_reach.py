"""The multi-layer reduction's skipping: layers in any order, chunks that only
some of the layers reach, rows and sources on the edges of chunks and row
blocks, and coordinates that are not numbers. Skipping leaves every bit as it
is, so the sums with and without it are compared bitwise; the values against
the oracle within the matvec tolerance (2e-5 of the sum of absolute terms)."""
import numpy as np
import pytest

from paper_2105_09465_gb300 import abi, api, workloads as W
from tests.gpu_util import assert_matvec_close, dev, host, need_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    need_gpu()


@pytest.mark.parametrize("L,nrhs,n,side", [(1, 1, 1, (1, 1)), (2, 1, 255, (9, 5)), (3, 4, 257, (63, 33)),
                                           (4, 2, 513, (64, 32)), (4, 4, 2049, (65, 31)), (3, 3, 4100, (40, 40))])
def test_layers_in_any_order_and_partial_reach(orc, L, nrhs, n, side):
    rng = np.random.default_rng(100 * L + nrhs)
    g = W.Grid(side[0], side[1], 1, 0.05)
    x = rng.uniform(-1.6, 1.6, (n, 2)).astype(np.float32)
    y = orc.grid_points(*g.astuple())
    v = rng.standard_normal((L, g.n, nrhs)).astype(np.float32)
    # reaches from 0.04 to 2.7 arcsec, the widest neither first nor last
    ls = list(np.float32([0.05, 0.2, 0.003, 0.011][:L]))
    vs = list(np.float32([1.0, -0.7, 1.3, 0.4][:L]))
    for src in (api.Points(grid=g), api.Points(xy=dev(y))):
        got = host(api.gp_kernel_matvec_layers(api.Points(xy=dev(x)), src, dev(v), ls, vs))
        abi.load().lr_set_pair_culling(0)
        try:
            full = host(api.gp_kernel_matvec_layers(api.Points(xy=dev(x)), src, dev(v), ls, vs))
        finally:
            abi.load().lr_set_pair_culling(1)
        assert np.array_equal(got, full)
        for h in range(nrhs):
            ref, ab = np.zeros(n), np.zeros(n)
            for k in range(L):
                o, a = orc.kernel_matvec(x, y, np.ascontiguousarray(v[k, :, h]), float(ls[k]), float(vs[k]))
                ref, ab = ref + o, ab + np.abs(a)
            assert_matvec_close(got[:, h], ref, ab, what=f"{L} layers, right-hand side {h}")


def test_a_row_that_is_not_a_number():
    g = W.Grid(40, 30, 1, 0.05)
    v = np.random.default_rng(3).standard_normal((2, g.n)).astype(np.float32)
    x = np.random.default_rng(4).uniform(-0.5, 0.5, (300, 2)).astype(np.float32)
    clean = host(api.gp_kernel_matvec_layers(api.Points(xy=dev(x)), api.Points(grid=g), dev(v), [0.05, 0.02],
                                             [1.0, 1.0]))
    x[128:256, 0] = np.nan  # a whole warp's rows among them
    out = host(api.gp_kernel_matvec_layers(api.Points(xy=dev(x)), api.Points(grid=g), dev(v), [0.05, 0.02],
                                           [1.0, 1.0]))
    assert np.isnan(out[128:256]).all() and np.isfinite(out[:128]).all() and np.isfinite(out[256:]).all()
    np.testing.assert_allclose(out[:128], clean[:128], rtol=0, atol=2e-5 * np.abs(v).sum(1).max())
