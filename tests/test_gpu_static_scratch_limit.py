"""gp_kernel_matvec_static_scratch just above its scratch: a sweep in parts whose
partial sums do not fit runs with one CTA per block of rows. Values against the
FP64 oracle on sampled rows within the matvec tolerance, the same bits at every
call, and within the rounding of the call with a workspace."""
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


def test_without_parts_where_they_do_not_fit(orc):
    lib = abi.load()
    cap = int(lib.lr_static_scratch_bytes())
    xg, nrhs, ell = W.Grid(300, 300, 1, 0.01), 4, 0.01
    q = api.Points(grid=xg)
    # the smallest source grid (by steps of 20) whose plan in parts is beyond the scratch
    side = next(k for k in range(400, 2000, 20)
                if api.matvec_workspace_size(q, api.Points(grid=W.Grid(k, k, 1, 3.2 / k)), nrhs) > cap)
    yg = W.Grid(side, side, 1, 3.2 / side)
    s = api.Points(grid=yg)
    v = np.random.default_rng(1).standard_normal((yg.n, nrhs)).astype(np.float32)
    tv = dev(v)
    cq, k1 = api.to_c_points(q)
    cs, k2 = api.to_c_points(s)
    outs = []
    for _ in range(2):
        out = torch.full((xg.n, nrhs), 1e30, dtype=torch.float32, device="cuda")
        st = lib.gp_kernel_matvec_static_scratch(ctypes.byref(cq), ctypes.byref(cs), tv.data_ptr(), nrhs, ell, 1.0,
                                                 out.data_ptr(), None, torch.cuda.current_stream().cuda_stream)
        abi.check(st, "gp_kernel_matvec_static_scratch")
        outs.append(out)
    torch.cuda.synchronize()
    assert torch.equal(outs[0], outs[1])
    ref = api.gp_kernel_matvec(q, s, tv, ell)
    rows = np.random.default_rng(2).choice(xg.n, 60, replace=False)
    x, y = orc.grid_points(*xg.astuple()), orc.grid_points(*yg.astuple())
    for h in range(nrhs):
        want, ab = orc.kernel_matvec(x, y, v[:, h], ell, 1.0, rows=rows)
        for got in (outs[0], ref):
            assert_matvec_close(host(got)[rows, h], want, ab, what=f"right-hand side {h}")
