"""The multi-layer reduction over values that are not finite. Every row's sum
takes in every source: a weight that is not finite, or a source coordinate that
is not a number, makes every row of its right-hand side not a number, however far
the source (0 * inf, NaN * 0). A coordinate at infinity is only far. The values against the oracle within the matvec tolerance (2e-5 of the sum of
absolute terms)."""
import numpy as np
import pytest

from paper_2105_09465_gb300 import abi, api, workloads as W
from tests.gpu_util import assert_matvec_close, dev, host, need_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    need_gpu()


def layers(x, src, v, ls, vs, cull):
    abi.load().lr_set_pair_culling(cull)
    try:
        return host(api.gp_kernel_matvec_layers(api.Points(xy=dev(x)), src, dev(v), ls, vs))
    finally:
        abi.load().lr_set_pair_culling(1)


@pytest.mark.parametrize("what", ["weight nan", "weight inf", "source nan", "whole chunk nan"])
@pytest.mark.parametrize("cull", [1, 0])
# all pairs, the culled sweep in parts, and (above the waves for them) one CTA per row block
@pytest.mark.parametrize("n", [5, 700, 100000, 1000000])
def test_not_finite_reaches_every_row(what, cull, n):
    rng = np.random.default_rng(n)
    m = 2000
    x = rng.uniform(-1, 1, (n, 2)).astype(np.float32)
    y = rng.uniform(-1, 1, (m, 2)).astype(np.float32)
    y[64:96] += 500.0  # the chunk in question: out of every row's reach
    v = rng.standard_normal((2, m, 2)).astype(np.float32)
    hs = slice(0, 2)  # the right-hand sides it reaches
    if what == "weight nan":
        v[0, 70, 1] = np.nan
        hs = slice(1, 2)
    elif what == "weight inf":
        v[1, 64, 0] = -np.inf
        hs = slice(0, 1)
    elif what == "source nan":
        y[95, 1] = np.nan
    else:
        y[64:96] = np.nan
    out = layers(x, api.Points(xy=dev(y)), v, [0.05, 0.02], [1.0, 0.5], cull)
    assert np.isnan(out[:, hs]).all()
    if hs != slice(0, 2):
        assert np.isfinite(np.delete(out, hs, axis=1)).all()


@pytest.mark.parametrize("n", [5, 700])
def test_infinite_coordinates_are_out_of_reach(orc, n):
    """A source at infinity has kernel value 0, a query there sees nothing."""
    rng = np.random.default_rng(n)
    x = rng.uniform(-1, 1, (n, 2)).astype(np.float32)
    y = rng.uniform(-1, 1, (300, 2)).astype(np.float32)
    v = rng.standard_normal((2, 300)).astype(np.float32)
    ls, vs = [0.3, 0.1], [1.0, 0.5]
    y[33, 0] = np.inf
    x[n - 1, 1] = -np.inf
    out = layers(x, api.Points(xy=dev(y)), v, ls, vs, 1)
    assert out[n - 1] == 0.0
    keep = np.arange(300) != 33
    ref, ab = np.zeros(n - 1), np.zeros(n - 1)
    for k in range(2):
        o, a = orc.kernel_matvec(x[:-1], y[keep], np.ascontiguousarray(v[k, keep]), ls[k], vs[k])
        ref, ab = ref + o, ab + np.abs(a)
    assert_matvec_close(out[:-1], ref, ab, what="infinite source")
