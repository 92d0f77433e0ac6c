"""Subhalo records at the edges of what a fit or a padded list holds, where
tiles take the local expansion: zero mass (kappa_s = 0: the deflection is 0 but
its derivative by kappa_s is not), a negative scale radius (only its square and
its modulus enter), and coordinates far from the size of an arcsecond. Values
against the FP64 oracle: gradients within 2e-5 of the sum of absolute terms
(the repository's gradient tolerance), deflections within 1e-6 of the scale of
the coordinates."""
import numpy as np
import pytest

from paper_2105_09465_gb300 import api, workloads as W
from tests.gpu_util import ALPHA_TOL, GRAD_REL, assert_close_tol, dev, host, need_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    need_gpu()


def check_vjp(orc, g, lens, sub, d, ref_sub=None, sign=1.0):
    """Subhalo gradients of the grid g against the oracle's for ref_sub, its
    theta_s column times sign."""
    xi = orc.grid_points(*g.astuple())
    _, ds = api.lens_raytrace_vjp(api.Points(grid=g, lens=lens, sub=dev(sub)), dev(d))
    _, rs, _, asub = orc.raytrace_vjp(xi.astype(np.float64), lens.astuple(), sub if ref_sub is None else ref_sub,
                                      d.astype(np.float64), with_abs=True)
    rs[:, 3] *= sign
    assert np.isfinite(host(ds)).all()
    assert_close_tol(host(ds), rs, GRAD_REL * asub, what="subhalos")


def population(rng, n_sub):
    """Near and far subhalos of a field of about 4 arcsec."""
    return np.column_stack([rng.uniform(-9, 9, (n_sub, 2)), rng.uniform(0.01, 0.1, n_sub),
                            rng.uniform(0.02, 0.1, n_sub), rng.uniform(1, 15, n_sub)]).astype(np.float32)


# 640k points x 200: more than one wave of tiles, ordered by the plan
@pytest.mark.parametrize("n_sub,side,which", [(1, 32, "all"), (17, 32, "one"), (17, 32, "all"), (200, 32, "one"),
                                              (200, 32, "half"), (200, 32, "all"), (257, 60, "half"),
                                              (200, 400, "half")])
def test_zero_mass(orc, n_sub, side, which):
    rng = np.random.default_rng(n_sub + side)
    g = W.Grid(side, side, 2, 4.0 / side)
    sub = population(rng, n_sub)
    sub[{"one": slice(0, 1), "half": slice(n_sub // 2, None), "all": slice(None)}[which], 2] = 0.0
    check_vjp(orc, g, W.draw_lens(rng), sub, rng.standard_normal((g.n, 2)).astype(np.float32))


@pytest.mark.parametrize("n_sub", [17, 200])
def test_negative_scale_radius_backward(orc, n_sub):
    rng = np.random.default_rng(n_sub)
    ref = population(rng, n_sub)
    ref[:, :2] /= 3.0
    ref[:, 3:] = (0.1, 1.0)  # the series' odd terms: 7e-4 of the sums at 1.6 arcsec
    sub = ref.copy()
    sub[:, 3] *= -1.0
    g = W.Grid(40, 40, 2, 0.02)  # 50 tiles of 8 x 16 points
    # one gradient at every point: the sums are of the size of their absolute terms
    check_vjp(orc, g, W.draw_lens(rng), sub, np.tile(np.float32([0.8, -0.6]), (g.n, 1)), ref, -1.0)


@pytest.mark.parametrize("n_sub", [64, 300])
def test_negative_scale_radius_forward(orc, n_sub):
    g = W.Grid(90, 33, 2, 0.01)
    lens = W.Lens(0.0, 0.0, 0.9, 0.2, 1e-9, 2.0, 0.0, 0.0)
    rng = np.random.default_rng(n_sub)
    ref = population(rng, n_sub)
    ref[:, 2:] = (6.0 / n_sub, 0.1, 1.0)
    t = rng.uniform(0, 2 * np.pi, n_sub)  # the odd terms are 3e-4 of the deflection, 0.03 arcsec
    ref[:, 0], ref[:, 1] = 2.15 + 0.05 * np.cos(t), 0.05 * np.sin(t)
    sub = ref.copy()
    sub[:, 3] *= -1.0
    _, alpha = api.lens_raytrace(api.Points(grid=g, lens=lens, sub=dev(sub)), want_alpha=True)
    want, _ = orc.raytrace(orc.grid_points(*g.astuple()), lens.astuple(), ref, 0)
    assert np.abs(host(alpha) - want).max() <= ALPHA_TOL


@pytest.mark.parametrize("scale", [2.0**-18, 2.0**18])
@pytest.mark.parametrize("n_sub", [17, 200])
def test_scale_of_the_coordinates(orc, n_sub, scale):
    rng = np.random.default_rng(n_sub)
    g = W.Grid(90, 33, 2, 0.05 * scale)
    lens = W.Lens(0.0, 0.0, 0.9, 0.2, 1e-9 * scale, 2.0, 0.0, 0.0)
    sub = population(rng, n_sub)
    sub[:, [0, 1, 3]] *= np.float32(scale)
    check_vjp(orc, g, lens, sub, rng.standard_normal((g.n, 2)).astype(np.float32))
    _, alpha = api.lens_raytrace(api.Points(grid=g, lens=lens, sub=dev(sub)), want_alpha=True)
    want, _ = orc.raytrace(orc.grid_points(*g.astuple()), lens.astuple(), sub, 0)
    assert np.abs(host(alpha) - want).max() <= ALPHA_TOL * scale
