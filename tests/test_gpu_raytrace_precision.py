"""Precision of the far subhalos' sum by a grid tile's local expansion. All
subhalos lie to one side, so that the deflection is of the size of the sum of its
absolute terms, and the main lens deflects by 1e-9 arcsec.

Against the direct sums of the same points handed over as a list: the errors'
spread over the points may exceed the direct sums' by a tenth at most. (Their
mean is left out: the records' FP32 constants shift every point of both by the
same, and the direct sums' series of the fewest terms by some 1e-8 more.)

With masses that cancel: the sums over the first two of the CTA's four warps (or
the first two of four windows of 2048 subhalos) and over the last two are exact
negatives, so the total is 0 but for what the additions between them round away.
The constant term's additions are compensated; the other terms, at most 0.037 of
it here (a half-diagonal of 0.133 arcsec at 3.6), are added plainly: three
roundings of 2^-24 of them, 7e-9 of the sum of absolute terms."""
import numpy as np
import pytest

from paper_2105_09465_gb300 import api, workloads as W
from tests.gpu_util import dev, host, need_gpu

pytestmark = pytest.mark.gpu

GRID = W.Grid(80, 16, 2, 0.025)
LENS = W.Lens(0.0, 0.0, 0.9, 0.2, 1e-9, 2.0, 0.0, 0.0)


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    need_gpu()


def population(n_sub, lo, hi, tau):
    rng = np.random.default_rng(n_sub)
    return np.column_stack([rng.uniform(lo, hi, n_sub), rng.uniform(-4, 4, n_sub),
                            rng.uniform(0.01, 0.1, n_sub) * 200 / n_sub, rng.uniform(0.01, 0.1, n_sub),
                            rng.uniform(1, tau, n_sub)]).astype(np.float32)


def error(orc, sub, **points):
    ref, _ = orc.raytrace(orc.grid_points(*GRID.astuple()), LENS.astuple(), sub, 0)
    _, alpha = api.lens_raytrace(api.Points(lens=LENS, sub=dev(sub), **points), want_alpha=True)
    return host(alpha) - ref


@pytest.mark.parametrize("lo,hi,tau", [(4.0, 12.0, 2.0), (4.0, 12.0, 15.0), (40.0, 60.0, 15.0)])
@pytest.mark.parametrize("n_sub", [64, 129, 2048, 4097])
def test_spread_against_the_direct_sums(orc, n_sub, lo, hi, tau):
    sub = population(n_sub, lo, hi, tau)
    far = error(orc, sub, grid=GRID)[:, 0].std()
    direct = error(orc, sub, xy=dev(orc.grid_points(*GRID.astuple())))[:, 0].std()
    assert far <= 1.1 * direct, f"expansion {far:.3e}, direct sums {direct:.3e} arcsec"


@pytest.mark.parametrize("n_sub", [128, 8192])
def test_cancelling_masses(orc, n_sub):
    sub = population(n_sub, 4.0, 12.0, 2.0)
    half = n_sub // 2
    sub[half:] = sub[:half]
    sub[half:, 2] *= -1.0
    xi = orc.grid_points(*GRID.astuple())
    scale = 2.0 * np.abs(orc.raytrace(xi, LENS.astuple(), sub[:half], 0)[0][:, 0]).max()
    err = np.abs(error(orc, sub, grid=GRID)).max()
    assert err <= 7e-9 * scale, f"{err / scale:.3e} of the sum of absolute terms"
