"""Small ray-traces (one wave of CTAs of 256 threads, one point each) against
larger ones (two points per thread): a point list and the same list with more
points after it are traced in the same tiles, so the common points have the
same bits. Sizes: one point, a ragged tile, a few tiles, near the largest that
fits; staged chunks of subhalos whole, ragged and several.
"""
import numpy as np
import pytest
import torch

from paper_2105_09465_gb300 import api, workloads as W
from tests.gpu_util import dev, need_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    need_gpu()


@pytest.mark.parametrize("profile", [0, 1])
@pytest.mark.parametrize("n,n_sub", [(1, 1), (255, 3), (257, 64), (5000, 256), (5000, 257), (110_000, 601)])
def test_small_bits(profile, n, n_sub):
    rng = np.random.default_rng(11)
    xy = rng.uniform(-4, 4, (200_000, 2)).astype(np.float32)
    xy[:n] = xy[:n][np.lexsort(xy[:n].T)]
    lens = W.Lens(0.02, -0.01, 0.8, 0.3, 1.1, 2.1, 0.02, -0.01)
    sub = np.column_stack([rng.uniform(-4, 4, (n_sub, 2)), rng.uniform(0.01, 0.05, (n_sub, 2)),
                           rng.uniform(1, 15, n_sub)]).astype(np.float32)
    m = n // 256 * 256 if n >= 256 else n  # whole tiles, or the one tile's points alone
    big = api.lens_raytrace(api.Points(xy=dev(xy), lens=lens, sub=dev(sub), profile=profile))
    small = api.lens_raytrace(api.Points(xy=dev(xy[:n]), lens=lens, sub=dev(sub), profile=profile))
    if n >= 256:
        assert torch.equal(small[:m], big[:m])
    else:  # the tile of the large call holds other points: its series may differ
        assert torch.allclose(small, big[:n], rtol=0, atol=1e-6)
