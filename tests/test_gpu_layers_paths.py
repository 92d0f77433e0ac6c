"""The multi-layer reduction's two paths (the sweep over all pairs for small
problems and for grids within every layer's reach, the culled chunk sweep for
the rest): the culled sweep at sizes that take it, with few and many rows, lists
and image layouts, on and off the edges of row blocks and chunks; and both sides
of either line of the rule. Sampled rows against the FP64 oracle within the
matvec tolerance (2e-5 of the sum of absolute terms); skipping leaves every bit as
it is."""
import numpy as np
import pytest

from paper_2105_09465_gb300 import abi, api, workloads as W
from tests.gpu_util import assert_matvec_close, dev, host, need_gpu

pytestmark = pytest.mark.gpu

SMALL = 3.5e8  # n m (1 + L + L nrhs) up to which every pair is formed


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    need_gpu()


def check(orc, q, x, src, y, v, ls, vs, what):
    """v (L, m, nrhs); every right-hand side on 40 rows, the last among them."""
    got = host(api.gp_kernel_matvec_layers(q, src, dev(v), ls, vs)).reshape(len(x), -1)
    abi.load().lr_set_pair_culling(0)
    try:
        full = host(api.gp_kernel_matvec_layers(q, src, dev(v), ls, vs)).reshape(len(x), -1)
    finally:
        abi.load().lr_set_pair_culling(1)
    assert np.array_equal(got, full)
    rows = np.unique(np.append(np.random.default_rng(7).integers(0, len(x), 39), len(x) - 1))
    for h in range(v.shape[2]):
        ref, ab = np.zeros(len(rows)), np.zeros(len(rows))
        for k in range(v.shape[0]):
            o, a = orc.kernel_matvec(x, y, np.ascontiguousarray(v[k, :, h]), float(ls[k]), float(vs[k]), rows=rows)
            ref, ab = ref + o, ab + np.abs(a)
        assert_matvec_close(got[rows, h], ref, ab, what=f"{what}, right-hand side {h}")


def hyper(L):
    return list(np.float32([0.05, 0.2, 0.003, 0.011][:L])), list(np.float32([1.0, -0.7, 1.3, 0.4][:L]))


@pytest.mark.parametrize("L,nrhs", [(1, 1), (2, 1), (4, 2), (3, 4)])
@pytest.mark.parametrize("n", [257, 2049, 30011])
def test_culled_lists(orc, L, nrhs, n):
    rng = np.random.default_rng(n + L)
    m = int(1.2 * SMALL / (n * (1 + L + L * nrhs))) + 1
    x = rng.uniform(-1.6, 1.6, (n, 2)).astype(np.float32)
    y = rng.uniform(-1.6, 1.6, (m, 2)).astype(np.float32)
    y = y[np.lexsort((y[:, 0], np.floor(y[:, 1] * 20)))]  # rows of sources: chunks that some layers do not reach
    v = rng.standard_normal((L, m, nrhs)).astype(np.float32)
    ls, vs = hyper(L)
    check(orc, api.Points(xy=dev(x)), x, api.Points(xy=dev(y)), y, v, ls, vs, "list")


@pytest.mark.parametrize("L,nrhs", [(1, 1), (3, 1), (2, 4)])  # 4 and 2 rows per thread
@pytest.mark.parametrize("side", [(64, 32), (70, 131), (201, 77)])
@pytest.mark.parametrize("query", ["grid", "lensed", "layout", "self"])
def test_culled_queries_in_an_image_layout(orc, L, nrhs, side, query):
    rng = np.random.default_rng(10 * L + side[0])
    if query == "self":
        side = (3 * side[0] + 1, 2 * side[1])
    g = W.Grid(side[0], side[1], 1, 3.0 / side[0])
    k = int(np.sqrt(1.2 * SMALL / (g.n * (1 + L + L * nrhs)))) + 1
    yg = W.Grid(k + 1, k, 1, 3.2 / k)
    src, y = api.Points(grid=yg), orc.grid_points(*yg.astuple())
    if query in ("grid", "self"):
        x, q = orc.grid_points(*g.astuple()), api.Points(grid=g)
    elif query == "lensed":
        q = api.Points(grid=g, lens=W.Lens(0.01, -0.02, 0.8, 0.3, 0.7, 2.0, 0.01, 0.0))
        x = host(api.lens_raytrace(q)).astype(np.float32)  # the library's own points, on both sides
    else:
        x = rng.uniform(-1.5, 1.5, (g.n, 2)).astype(np.float32)
        q = api.Points(xy=dev(x), grid=g)
    if query == "self":
        src, y = None, x
    v = rng.standard_normal((L, len(y), nrhs)).astype(np.float32)
    ls, vs = hyper(L)
    check(orc, q, x, src, y, v, ls, vs, f"{query} query")


@pytest.mark.parametrize("L,nrhs", [(1, 1), (3, 4)])
@pytest.mark.parametrize("factor", [0.999, 1.001])
def test_both_sides_of_the_size(orc, L, nrhs, factor):
    rng = np.random.default_rng(3)
    n = 3001
    m = int(factor * SMALL / (n * (1 + L + L * nrhs)))
    x, y = (rng.uniform(-1.6, 1.6, (k, 2)).astype(np.float32) for k in (n, m))
    v = rng.standard_normal((L, m, nrhs)).astype(np.float32)
    ls, vs = hyper(L)
    check(orc, api.Points(xy=dev(x)), x, api.Points(xy=dev(y)), y, v, ls, vs, f"{factor} of the size")


@pytest.mark.parametrize("own", [False, True])
@pytest.mark.parametrize("factor", [0.999, 1.001])
@pytest.mark.parametrize("L,nrhs", [(2, 1), (3, 4)])
def test_both_sides_of_the_reach(orc, L, nrhs, factor, own):
    """Grid sources, or a grid on itself, whose diagonal is factor times the
    narrowest layer's reach."""
    rng = np.random.default_rng(4)
    yg = W.Grid(131, 125, 1, 0.02) if own else W.Grid(257, 31, 1, 0.02)
    diag = 0.02 * np.hypot(yg.nx - 1, yg.ny - 1)
    narrow = diag / (factor * np.sqrt(2 * np.log(2) * 127.0))
    ls, vs = list(np.float32([1.7, 1.0, 1.3][:L]) * np.float32(narrow)), [1.0, -0.6, 0.8][:L]
    y = orc.grid_points(*yg.astuple())
    x = y if own else rng.uniform(-2, 2, (20000, 2)).astype(np.float32)
    v = rng.standard_normal((L, yg.n, nrhs)).astype(np.float32)
    q = api.Points(grid=yg) if own else api.Points(xy=dev(x))
    check(orc, q, x, None if own else api.Points(grid=yg), y, v, ls, vs, f"{factor} of the reach")
