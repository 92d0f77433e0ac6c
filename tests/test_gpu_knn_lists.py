"""The k-nearest-neighbour query's list lengths (k rounded up to a multiple of
four) and cell runs: every k on both sides of a rounding, the fewest points that
have a k-th other neighbour, points in one cell row or column, and the weights
of a second length scale from the same radii."""
import numpy as np
import pytest
import torch

from paper_2105_09465_gb300 import api
from tests.gpu_util import dev, host, need_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    need_gpu()


@pytest.mark.parametrize("k", [1, 3, 4, 5, 8, 9, 16, 19, 20, 21, 28, 31, 32])
@pytest.mark.parametrize("shape", ["least", "row", "column", "clustered"])
def test_every_list_length(orc, k, shape):
    rng = np.random.default_rng(k)
    if shape == "least":
        q = rng.uniform(-1, 1, (k + 1, 2))
    elif shape == "clustered":
        q = np.concatenate([rng.normal(0, 0.01, (400, 2)), rng.uniform(-2, 2, (301, 2))])
    else:
        q = np.stack([rng.uniform(-1, 1, 500), np.full(500, 0.25)], 1)
        q = q if shape == "row" else q[:, ::-1]
    q = np.ascontiguousarray(q, np.float32)
    r2, a = api.knn_density(dev(q), k, lengthscale=0.07)
    ref = orc.knn_r2(q, k)
    # FP32 squared distances of the same FP32 points: a few 2^-24 relative
    assert np.all(np.abs(host(r2) - ref) <= 1e-6 * ref)
    assert torch.equal(api.transmission_weights(r2, k, 0.07), a)
    _, b = api.knn_density(dev(q), k, lengthscale=0.013)
    assert torch.equal(api.transmission_weights(r2, k, 0.013), b)
