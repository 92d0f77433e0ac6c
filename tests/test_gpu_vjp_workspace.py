"""The ray-trace VJP's workspace: where every tile adds its own phases (tNFW,
at most 4096 subhalos, tiles within one staged chunk) it holds no slot sums, so it
grows with the subhalo count; point masses keep theirs. And the gradients at the
counts that used to take several phases per launch, in a workspace of exactly
that size, against the FP64 oracle."""
import ctypes

import numpy as np
import pytest
import torch

from paper_2105_09465_gb300 import abi, api, workloads as W
from tests.gpu_util import GRAD_REL, assert_close_tol, dev, host, need_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    need_gpu()


def size(points):
    c, keep = api.to_c_points(points)
    b = ctypes.c_size_t()
    abi.check(abi.load().lr_raytrace_vjp_workspace_size(ctypes.byref(c), ctypes.byref(b)), "size")
    return b.value


def points(side, n_sub, profile=0):
    rng = np.random.default_rng(n_sub)
    lens = W.draw_lens(rng)
    sub = W.draw_subhalos(rng, n_sub, lens, 1e7, 1e10)
    if profile:
        sub[:, 2] = 0.01
    return api.Points(grid=W.Grid(side, side, 2, 6.0 / side), lens=lens, sub=dev(sub), profile=profile), lens, sub


@pytest.mark.parametrize("side", [230, 400])
def test_no_slot_sums_where_tiles_add_their_own(side):
    sizes = [size(points(side, k)[0]) for k in (127, 150, 200, 255)]
    assert sizes == sorted(sizes) and sizes[-1] < 2 * sizes[0] + 4096
    assert size(points(side, 150, 1)[0]) > size(points(side, 150)[0])  # 2 phases at either side


@pytest.mark.parametrize("profile", [0, 1])
def test_gradients_in_that_workspace(orc, profile):
    q, lens, sub = points(230, 200, profile)
    need = size(q)
    ws = torch.full((need + 512,), 0x7F, dtype=torch.uint8, device="cuda")
    lo = -ws.data_ptr() % 256
    d = np.random.default_rng(1).standard_normal((q.grid.n, 2)).astype(np.float32)
    c, keep = api.to_c_points(q)
    dl = torch.empty(7, dtype=torch.float64, device="cuda")
    ds = torch.empty((200, 4), dtype=torch.float64, device="cuda")
    td = dev(d)
    st = abi.load().lens_raytrace_vjp(ctypes.byref(c), td.data_ptr(), dl.data_ptr(), ds.data_ptr(), ws.data_ptr() + lo,
                                      need, torch.cuda.current_stream().cuda_stream)
    abi.check(st, "lens_raytrace_vjp")
    torch.cuda.synchronize()
    assert (ws[:lo] == 0x7F).all() and (ws[lo + need:] == 0x7F).all()  # nothing beyond it is written
    xi = orc.grid_points(*q.grid.astuple()).astype(np.float64)
    rl, rs, al, asub = orc.raytrace_vjp(xi, lens.astuple(), sub, d.astype(np.float64), profile, with_abs=True)
    assert_close_tol(host(dl), rl, GRAD_REL * al, what="lens")
    if profile:
        assert_close_tol(host(ds)[:, :3], rs[:, :3], GRAD_REL * asub[:, :3], what="subhalos")
    else:
        assert_close_tol(host(ds), rs, GRAD_REL * asub, what="subhalos")
