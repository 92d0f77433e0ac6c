"""The windowed reduction over few sources: none (with its likelihood the model is
f_in alone; library entry only, the Python wrapper hands an empty tensor over as
NULL, which the entry refuses), and up to 512, where each row block is one CTA
instead of parts, against the FP64 oracle within 2e-5 of the sum of absolute
terms."""
import ctypes

import numpy as np
import pytest
import torch

from paper_2105_09465_gb300 import abi, api, workloads as W
from tests.gpu_util import assert_matvec_close, dev, host, need_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    need_gpu()


@pytest.mark.parametrize("cull", [1, 0])
@pytest.mark.parametrize("n,layout", [(1, None), (300, None), (600, (30, 20))])
def test_likelihood_over_no_sources(n, layout, cull):
    lib = abi.load()
    rng = np.random.default_rng(n)
    p, z = rng.uniform(-1, 1, (n, 2)), np.tile([0.01, 0.0, 0.01], (n, 1))
    f, data, sigma = rng.standard_normal(n), rng.standard_normal(n), 0.3
    src = abi.lr_points()
    some = torch.zeros(2, dtype=torch.float32, device="cuda")  # a real address; no point is read
    src.xy, src.n = some.data_ptr(), 0
    lay = ctypes.byref(abi.lr_grid(*W.Grid(layout[0], layout[1], 1, 0.05).astuple())) if layout else None
    need = ctypes.c_size_t()
    abi.check(lib.lr_windowed_workspace_size(n, lay, ctypes.byref(src), ctypes.byref(need)), "workspace")
    ws = torch.full((need.value + 256,), 0x7F, dtype=torch.uint8, device="cuda")
    base = (ws.data_ptr() + 255) // 256 * 256
    out, g = (torch.full((n,), 1e30, device="cuda") for _ in range(2))
    nll = torch.full((1,), 1e30, dtype=torch.float64, device="cuda")
    tp, tz, tf, td = dev(p), dev(z), dev(f), dev(data)
    lib.lr_set_pair_culling(cull)
    try:
        st = lib.gp_windowed_matvec_nll(tp.data_ptr(), tz.data_ptr(), n, lay, ctypes.byref(src), some.data_ptr(), 0.05,
                                        tf.data_ptr(), td.data_ptr(), sigma, out.data_ptr(), g.data_ptr(),
                                        nll.data_ptr(), base, need.value, torch.cuda.current_stream().cuda_stream)
    finally:
        lib.lr_set_pair_culling(1)
    abi.check(st, "gp_windowed_matvec_nll")
    torch.cuda.synchronize()
    f32, d32 = f.astype(np.float32).astype(np.float64), data.astype(np.float32).astype(np.float64)
    s = float(np.float32(sigma))
    assert torch.equal(out, tf)
    np.testing.assert_allclose(g.cpu().numpy(), (f32 - d32) / s**2, rtol=1e-6, atol=1e-6)
    want = 0.5 * np.sum(((f32 - d32) / s) ** 2) + n * (np.log(s) + 0.5 * np.log(2 * np.pi))
    np.testing.assert_allclose(nll.item(), want, rtol=1e-6, atol=1e-6)


@pytest.mark.parametrize("m", [1, 31, 512, 513])
@pytest.mark.parametrize("n,layout", [(1, None), (300, None), (5000, (100, 50))])
def test_few_sources(orc, n, m, layout):
    rng = np.random.default_rng(n + m)
    lay = W.Grid(layout[0], layout[1], 1, 0.02) if layout else None
    p = orc.grid_points(*lay.astuple()) if lay else rng.uniform(-1, 1, (n, 2)).astype(np.float32)
    a = rng.uniform(0.01, 0.05, (n, 2, 2))
    z = np.stack([(a[:, 0] * a[:, 0]).sum(1), (a[:, 0] * a[:, 1]).sum(1), (a[:, 1] * a[:, 1]).sum(1)], 1)
    z = z.astype(np.float32)
    q, v = rng.uniform(-1, 1, (m, 2)).astype(np.float32), rng.standard_normal(m).astype(np.float32)
    f, data = (rng.standard_normal(n).astype(np.float32) for _ in range(2))
    ell, sigma = 0.05, 0.3
    src = api.Points(xy=dev(q))
    ref, ab = orc.windowed_matvec(p, z, q, v, ell)
    got = api.gp_windowed_matvec(dev(p), dev(z), src, dev(v), ell, layout=lay)
    assert_matvec_close(host(got), ref, ab, what="windowed")
    out, g, nll = api.gp_windowed_matvec_nll(dev(p), dev(z), src, dev(v), ell, dev(data), sigma, f_in=dev(f), layout=lay)
    assert_matvec_close(host(out), ref + f, ab + np.abs(f), what="model")
    r = (host(out) - data) / np.float32(sigma)
    np.testing.assert_allclose(host(g), r / np.float32(sigma), rtol=1e-5, atol=1e-5)
    np.testing.assert_allclose(nll.item(), 0.5 * (r * r).sum() + n * (np.log(np.float64(np.float32(sigma)))
                                                                      + 0.5 * np.log(2 * np.pi)), rtol=1e-5, atol=1e-5)
