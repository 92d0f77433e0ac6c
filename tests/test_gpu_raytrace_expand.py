"""The forward ray-trace's local expansion of the far subhalos about a grid
tile's centre: on grids with rows of 160 points, where at least 40 + n_sub / 4
of at least 64 subhalos are 12.5 half-diagonals from it, those far from the
whole tile (and served by the series of degree 7) are summed as one polynomial
of 36 terms per tile; the rest are listed and summed directly.

Copies of one heavy subhalo at one distance at a time, on and off axis, with
the copy count at the edges of the rule (64), of a round of threads (128) and
of a window (2048). All deflections have one sign, so the relative bound of a
single subhalo's series holds for the sum, 1.5e-6 (ten FP32 roundings and the
2^-22.9 of the reciprocal square root), and up to 6e-7 more for a thread's
plain sum of 16 equal terms, which round alike, and the polynomial: 2.2e-6. A
dropped or wrong term of the expansion of relative size 1e-5 fails. Then a
random population over ragged grids, single rows and a last tile of one pixel,
within 1e-6 arcsec as every deflection.
"""
import numpy as np
import pytest

from paper_2105_09465_gb300 import api, workloads as W
from tests.gpu_util import dev, host, need_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    need_gpu()


# grid centres (arcsec): the 16 x 16 tiles' half-diagonals are 0.13 arcsec and
# the grid spans 1 arcsec to either side, so the first has tiles on either side
# of the limit of 1.7 arcsec, the rest are far
@pytest.mark.parametrize("cx,cy", [(2.2, 0.0), (2.5, -2.2), (-9.0, 4.0), (60.0, 45.0)])
@pytest.mark.parametrize("copies", [63, 64, 128, 129, 2048, 2049])
def test_expansion_relative(orc, copies, cx, cy):
    g = W.Grid(80, 9, 2, 0.025, cx, cy)
    lens = W.Lens(0.0, 0.0, 0.9, 0.2, 1e-9, 2.0, 0.0, 0.0)
    sub = np.repeat(np.array([[0.0, 0.0, 0.05, 0.02, 5.0]], np.float32), copies, axis=0)
    xi = orc.grid_points(*g.astuple())
    _, alpha = api.lens_raytrace(api.Points(grid=g, lens=lens, sub=dev(sub)), want_alpha=True)
    ref, _ = orc.raytrace(xi, lens.astuple(), sub, 0)
    err = np.hypot(*(host(alpha).astype(np.float64) - ref).T) / np.hypot(*ref.T)
    assert err.max() <= 2.2e-6, f"max relative deflection error {err.max():.3e}"


@pytest.mark.parametrize("nx,ny,ss,n_sub", [(177, 17, 1, 128), (83, 31, 2, 200), (1, 190, 1, 150), (159, 3, 1, 200),
                                             (161, 33, 1, 4097)])
def test_expansion_population(orc, nx, ny, ss, n_sub):
    rng = np.random.default_rng(7)
    g = W.Grid(nx, ny, ss, 0.05, 0.3, -0.2)
    lens = W.Lens(0.02, -0.01, 0.8, 0.3, 1.1, 2.1, 0.02, -0.01)
    sub = np.column_stack([rng.uniform(-9, 9, (n_sub, 2)), rng.uniform(0.01, 0.1, n_sub) * 200 / n_sub,
                           rng.uniform(0.01, 0.1, n_sub), rng.uniform(1, 15, n_sub)]).astype(np.float32)
    xi = orc.grid_points(*g.astuple())
    _, alpha = api.lens_raytrace(api.Points(grid=g, lens=lens, sub=dev(sub)), want_alpha=True)
    ref, _ = orc.raytrace(xi, lens.astuple(), sub, 0)
    assert np.abs(host(alpha).astype(np.float64) - ref).max() <= 1e-6
