"""The parameter gradients as one float32 array: values, zero slots, missing
inputs, and the autograd wrapper taking them for float32 device parameters and
the FP64 route for others, with the same values."""
import numpy as np
import pytest
import torch

from paper_2105_09465_gb300 import api, workloads as W
from paper_2105_09465_gb300.autograd import lensed_gp_matvec
from tests.gpu_util import dev, need_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    need_gpu()


@pytest.mark.parametrize("n_sub", [0, 1, 51, 700])
@pytest.mark.parametrize("missing", [(), ("lens",), ("lengthscale", "sub")])
def test_layout(n_sub, missing):
    g = torch.Generator(device="cuda").manual_seed(n_sub)
    r = lambda *s: torch.randn(s, dtype=torch.float64, device="cuda", generator=g)
    G = {"lens": r(7), "lengthscale": r(1), "variance": r(1), "sub": r(n_sub, 4)}
    G = {k: t for k, t in G.items() if k not in missing}
    out = api.param_grads(G, n_sub, torch.device("cuda"))
    ref = torch.zeros(12 + 5 * n_sub, device="cuda")
    if "lens" in G:
        ref[:5], ref[6:8] = G["lens"][:5].float(), G["lens"][5:].float()
    if "lengthscale" in G:
        ref[8] = G["lengthscale"][0].float()
    ref[9] = G["variance"][0].float()
    if "sub" in G:
        ref[12:].view(n_sub, 5)[:, :4] = G["sub"].float()
    assert torch.equal(out, ref)


@pytest.mark.parametrize("n_sub", [0, 7])
def test_wrapper_routes_agree(n_sub):
    p = W.realistic(seed=9, side=24, ss=2, n_sub=n_sub)
    g = dev(np.random.default_rng(1).standard_normal(p.n))
    grads = []
    for dtype, where in ((torch.float32, "cuda"), (torch.float64, "cuda"), (torch.float32, "cpu")):
        leaf = lambda a: torch.tensor(a, dtype=torch.float32).to(where, dtype).requires_grad_()
        v = dev(p.v).requires_grad_()
        sub = dev(p.sub).requires_grad_() if n_sub else None
        t = [v, leaf(list(p.lens.astuple())), leaf(p.lengthscale), leaf([1.0]).reshape(()).detach().requires_grad_()]
        lensed_gp_matvec(t[0], t[1], sub, t[2], t[3], p.xgrid, p.ygrid).backward(g)
        ts = t + ([sub] if n_sub else [])
        assert all(a.grad.shape == a.shape and a.grad.dtype == a.dtype and a.grad.device == a.device for a in ts)
        grads.append([a.grad.to("cuda", torch.float32) for a in ts])
    for other in grads[1:]:
        assert all(torch.equal(a, b) for a, b in zip(grads[0], other))
