"""Entries that run two branches side by side (the windowed backward, the grid
backward with saved moments) with several callers: threads on their own
streams, a capture beside an eager call of another thread or of the same one,
and more streams than the library keeps side streams for (16). Every result is
compared bit for bit with a lone call's."""
import ctypes
import threading

import numpy as np
import pytest
import torch

from paper_2105_09465_gb300 import abi, api, workloads as W
from tests.gpu_util import dev, need_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    need_gpu()


def windowed(seed):
    rng = np.random.default_rng(seed)
    n, m = 3000, 2500
    p, q = dev(rng.uniform(-1, 1, (n, 2))), dev(rng.uniform(-1, 1, (m, 2)))
    z = dev(np.tile([0.002, 0.0005, 0.001], (n, 1)))
    v, g = dev(rng.standard_normal(m)), dev(rng.standard_normal(n))
    return lambda: api.gp_windowed_matvec_bwd(p, z, api.Points(xy=q), v, 0.05, g)


def grid(seed):
    p = W.realistic(seed=seed, side=40, ss=2, n_sub=20)
    q = api.Points(grid=p.xgrid, lens=p.lens, sub=dev(p.sub))
    s = api.Points(grid=p.ygrid)
    v = dev(p.v)
    g = dev(np.random.default_rng(seed).standard_normal(p.xgrid.n))
    beta = torch.empty((p.xgrid.n, 2), dtype=torch.float32, device="cuda")
    _, mom = api.gp_kernel_matvec_train(q, s, v, p.lengthscale, p.variance, beta=beta)
    return lambda: api.gp_kernel_matvec_bwd(q, s, v, p.lengthscale, p.variance, g, beta=beta, moments=mom,
                                            want=("v", "lens", "sub", "lengthscale", "variance"))


def windowed_in_place(seed):
    """The same through the library entry, into buffers that exist (PyTorch's
    allocator may not grow in the thread that captures)."""
    rng = np.random.default_rng(seed)
    n, m = 3000, 2500
    p, q = dev(rng.uniform(-1, 1, (n, 2))), dev(rng.uniform(-1, 1, (m, 2)))
    z = dev(np.tile([0.002, 0.0005, 0.001], (n, 1)))
    v, g = dev(rng.standard_normal(m)), dev(rng.standard_normal(n))
    src, keep = api.to_c_points(api.Points(xy=q))
    need = ctypes.c_size_t()
    lib = abi.load()
    abi.check(lib.lr_windowed_bwd_workspace_size(n, None, ctypes.byref(src), ctypes.byref(need)), "workspace")
    ws = torch.empty(need.value, dtype=torch.uint8, device="cuda")
    out = {"v": torch.empty(m, device="cuda"), "p": torch.empty((n, 2), device="cuda"),
           "q": torch.empty((m, 2), device="cuda"), "z": torch.empty((n, 3), device="cuda"),
           "l": torch.empty(1, dtype=torch.float64, device="cuda")}

    def call():
        abi.check(lib.gp_windowed_matvec_bwd(p.data_ptr(), z.data_ptr(), n, None, ctypes.byref(src), v.data_ptr(),
                                             0.05, g.data_ptr(), *(out[k].data_ptr() for k in "vpqzl"), ws.data_ptr(),
                                             need.value, torch.cuda.current_stream().cuda_stream),
                  "gp_windowed_matvec_bwd")
        return out

    call.keep = (p, q, z, v, g, src, keep)
    return call


def same(a, b):
    return all(torch.equal(a[k], b[k]) for k in b)


def lone(fn):
    out = fn()
    torch.cuda.synchronize()
    return {k: t.clone() for k, t in out.items()}


@pytest.mark.parametrize("case", [windowed, grid])
def test_threads_on_their_own_streams(case):
    fns = [case(seed) for seed in range(4)]
    refs = [lone(f) for f in fns]
    bad = []

    def run(f, ref):
        s = torch.cuda.Stream()
        with torch.cuda.stream(s):
            for _ in range(20):
                out = f()
                s.synchronize()
                if not same(out, ref):
                    bad.append(1)

    ts = [threading.Thread(target=run, args=a) for a in zip(fns, refs)]
    [t.start() for t in ts]
    [t.join() for t in ts]
    assert not bad


@pytest.mark.parametrize("case", [windowed, grid])
def test_eager_call_of_another_thread_beside_a_capture(case):
    fa, fb = case(11), case(12)
    ra, rb = lone(fa), lone(fb)
    sa, sb = torch.cuda.Stream(), torch.cuda.Stream()
    got, err = {}, []

    def eager():
        try:
            with torch.cuda.stream(sb):
                got.update(fb())
            sb.synchronize()
        except Exception as e:  # reported below: an assertion here would end this thread alone
            err.append(e)

    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=sa, capture_error_mode="thread_local"):
        out = fa()
        t = threading.Thread(target=eager)
        t.start()
        t.join()
        out2 = fa()  # the capture goes on
    torch.cuda.synchronize()
    assert not err, err
    assert same(got, rb)
    for k in (out, out2):
        for t in k.values():
            t.zero_()
    graph.replay()
    torch.cuda.synchronize()
    assert same(out, ra) and same(out2, ra)


def test_eager_call_of_the_same_thread_beside_a_capture():
    fa, fb = windowed_in_place(11), windowed_in_place(12)
    ra, rb = lone(fa), lone(fb)
    sa, sb = torch.cuda.Stream(), torch.cuda.Stream()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=sa, capture_error_mode="thread_local"):
        fa()
        with torch.cuda.stream(sb):
            got = fb()
    torch.cuda.synchronize()
    assert same(got, rb)
    out = fa()  # the captured call's buffers
    for t in out.values():
        t.zero_()
    graph.replay()
    torch.cuda.synchronize()
    assert same(out, ra)
    for t in got.values():
        t.zero_()
    torch.cuda.synchronize()
    with torch.cuda.stream(sb):  # and after the capture
        fb()
    torch.cuda.synchronize()
    assert same(got, rb)


def test_more_streams_than_side_streams():
    f = windowed(3)
    ref = lone(f)
    outs = []
    streams = [torch.cuda.Stream(priority=k % 2 * -1) for k in range(40)]
    for s in streams:
        with torch.cuda.stream(s):
            outs.append(f())
    torch.cuda.synchronize()
    assert all(same(o, ref) for o in outs)
