"""The performance cases of this framework: the work its users have it do, through
the public entry points (`api`, `autograd`, `svi`, `serving`), at sizes from the
smallest calls to the largest configuration that one GPU holds.

A case is a dict of plain values with a `kind`:
  train        one training step of a lens system: fused ray-trace + kernel
               reduction, the Gaussian likelihood, and the whole backward
               (autograd); sources are a grid of inducing points or the
               ray-traced points themselves
  predict      the image of a drawn model: ray-trace + reduction, no gradients
  reconstruct  the source on a fine source-plane grid, several draws at once
  layers       several kernel layers sharing the pair distances, 1 or 4 draws
  raytrace     the lens alone (a user's own source model sits on top): rays of a
               masked pixel list, and the gradients of the lens and subhalos
  windowed     one image-plane layer: pixel windows, the windowed reduction of
               the ray-traced pixels against themselves, and its whole backward
  density      inducing-point densities and transmission weights (k = 20)
  svi          one variational-inference step of the paper's model
  serve        a batch of requests through the serving engine, host to host

Parameters live in float32 on the device, and their gradients are handed on in
the parameters' type, as an optimiser takes them.
"""
import math

import numpy as np
import torch

from paper_2105_09465_gb300 import api, svi
from paper_2105_09465_gb300.autograd import lensed_gp_matvec
from paper_2105_09465_gb300.serving import Session
from paper_2105_09465_gb300.workloads import Grid, Problem, draw_lens, draw_subhalos, draw_v, inducing_grid

# The paper's image-plane layers: kernel sizes (arcsec) and amplitudes.
SIGMA_LAYERS = (0.01, 0.00447213595499958, 0.002)
ALPHA_LAYERS = (0.3813263773918152, 0.19807367026805878, 0.15156535804271698)


def listed():
    return [
        # the smallest fit: a 100 x 100 cutout, the pixels as their own inducing
        # points, no subhalos: a step is a few small launches
        dict(name="fit_small", kind="train", source="self", nx=100, ny=100, ss=1, pix=0.05, n_sub=0, ell=0.05),
        # the paper's initial fit: 400 x 400 pixels of 12.5 mas against a
        # 40 x 40 source grid of 30 mas (the stationary kernel of 40 mas / sqrt 2)
        dict(name="fit_initial", kind="train", source="grid", nx=400, ny=400, ss=1, pix=0.0125, n_sub=0, side=40,
             src_pix=0.03, ell=0.0282842712),
        # a survey lens with substructure: 2 x 2 supersampling, 200 subhalos, 128 x 128 inducing points
        dict(name="fit_subhalos", kind="train", source="grid", nx=400, ny=400, ss=2, pix=0.05, n_sub=200, side=128,
             src_pix=0.0, ell=0.0),
        # the largest system: 2.56M points as their own inducing points, 2000 subhalos
        dict(name="fit_large", kind="train", source="self", nx=800, ny=800, ss=2, pix=0.05, n_sub=2000, ell=0.05),
        # posterior prediction of one image, an odd-sized cutout
        dict(name="predict_image", kind="predict", nx=331, ny=287, ss=2, pix=0.05, n_sub=150, side=128),
        # source reconstruction: 4 draws of the image-plane weights on a fine source-plane grid
        dict(name="reconstruct", kind="reconstruct", nx=400, ny=400, pix=0.05, n_sub=50, out=400, fov=4.0, nrhs=4,
             ell=0.05),
        # three layers on an inducing grid, 4 draws in one pass
        dict(name="layers_draws", kind="layers", nx=200, ny=200, ss=2, pix=0.05, n_sub=200, side=128, layers=3,
             nrhs=4),
        # a masked arc (odd pixel list, no image layout) through a lens with 500 subhalos
        dict(name="lens_masked", kind="raytrace", nx=389, ny=389, pix=0.025, r_in=0.4, r_out=4.6, n_sub=500),
        # the paper's widest image-plane layer
        dict(name="image_layer", kind="windowed", nx=400, ny=400, pix=0.0125, ell=SIGMA_LAYERS[0]),
        # transmission weights of a supersampled image's inducing points
        dict(name="density", kind="density", nx=800, ny=800, pix=0.025, n_sub=50, k=20, ell=0.05),
        # one SVI step of the paper's model: source-plane layer + three image-plane layers
        dict(name="svi_step", kind="svi", nx=400, ny=400, pix=0.0125, side=40, src_pix=0.03, sigma_sp=0.04, layers=3),
        # a serving batch: 4 requests of 64 to 256 px at 2 x 2, 10 iterations each
        dict(name="serve_batch", kind="serve", requests=4, side_lo=64, side_hi=256, max_sub=500, iters=10),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _ilog(rng, lo, hi):
    return int(round(_log(rng, lo, hi)))


def draw(rng):
    kind = rng.choice(["train", "train", "train", "predict", "reconstruct", "layers", "raytrace", "windowed",
                       "density", "svi", "serve"])
    c = dict(kind=kind)
    n_sub = 0 if rng.random() < 0.2 else _ilog(rng, 4, 500)
    if kind == "train":
        if rng.random() < 0.5:
            ss = rng.choice([1, 2])
            nx = _ilog(rng, 40, 640)
            c.update(source="self", nx=nx, ny=max(17, int(nx * rng.uniform(0.7, 1.0))), ss=ss, pix=0.05,
                     n_sub=min(n_sub * rng.choice([1, 2, 4]), 2000), ell=round(rng.uniform(0.04, 0.06), 4))
        elif rng.random() < 0.4:
            nx, sp = _ilog(rng, 64, 500), round(rng.uniform(0.02, 0.04), 4)
            c.update(source="grid", nx=nx, ny=max(31, int(nx * rng.uniform(0.7, 1.0))), ss=1, pix=0.0125, n_sub=0,
                     side=rng.randrange(30, 61), src_pix=sp, ell=round(sp * 0.942809, 6))
        else:
            nx = _ilog(rng, 48, 400)
            c.update(source="grid", nx=nx, ny=max(31, int(nx * rng.uniform(0.7, 1.0))), ss=2, pix=0.05, n_sub=n_sub,
                     side=rng.randrange(48, 129), src_pix=0.0, ell=0.0)
    elif kind == "predict":
        nx = _ilog(rng, 48, 420)
        c.update(nx=nx, ny=max(31, int(nx * rng.uniform(0.7, 1.0))), ss=rng.choice([1, 2]), pix=0.05, n_sub=n_sub,
                 side=rng.randrange(48, 129))
    elif kind == "reconstruct":
        nx = _ilog(rng, 60, 400)
        c.update(nx=nx, ny=max(31, int(nx * rng.uniform(0.7, 1.0))), pix=0.05, n_sub=n_sub // 4,
                 out=_ilog(rng, 64, 400), fov=4.0, nrhs=rng.choice([1, 2, 3, 4]), ell=0.05)
    elif kind == "layers":
        nx = _ilog(rng, 32, 200)
        c.update(nx=nx, ny=max(31, int(nx * rng.uniform(0.7, 1.0))), ss=2, pix=0.05, n_sub=n_sub,
                 side=rng.randrange(48, 129), layers=rng.choice([2, 3]), nrhs=rng.choice([1, 4]))
    elif kind == "raytrace":
        nx = _ilog(rng, 64, 420)
        fov = nx * 0.025
        c.update(nx=nx, ny=nx, pix=0.025, r_in=round(fov * rng.uniform(0.0, 0.1), 4),
                 r_out=round(fov * rng.uniform(0.35, 0.6), 4), n_sub=max(n_sub, 1))
    elif kind == "windowed":
        nx = _ilog(rng, 48, 400)
        c.update(nx=nx, ny=max(31, int(nx * rng.uniform(0.7, 1.0))), pix=0.0125, ell=round(_log(rng, 0.002, 0.02), 5))
    elif kind == "density":
        nx = _ilog(rng, 64, 800)
        c.update(nx=nx, ny=max(31, int(nx * rng.uniform(0.7, 1.0))), pix=0.025, n_sub=n_sub // 4,
                 k=20, ell=0.05)
    elif kind == "svi":
        nx = _ilog(rng, 64, 360)
        c.update(nx=nx, ny=max(31, int(nx * rng.uniform(0.7, 1.0))), pix=0.0125, side=rng.randrange(30, 51),
                 src_pix=0.03, sigma_sp=0.04, layers=rng.choice([1, 2, 3]))
    else:
        hi = rng.choice([96, 128, 192, 256])
        c.update(requests=rng.randrange(1, 6), side_lo=48, side_hi=hi, max_sub=500, iters=rng.randrange(2, 11))
    return c


# ---------------------------------------------------------------- inputs
def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a, np.float32)).cuda()


def _rng(case, seed):
    return np.random.default_rng([int(seed) % (1 << 32), 2105])


def _grid(c):
    return Grid(c["nx"], c["ny"], c.get("ss", 1), c["pix"])


def _lens(rng, c):
    """The survey priors, scaled down where the field is too small to hold the arcs."""
    lens = draw_lens(rng)
    room = 0.3 * min(c["nx"], c["ny"]) * c["pix"]
    if lens.theta_e > room:
        lens = type(lens)(**{**lens.asdict(), "theta_e": float(np.float32(room))})
    return lens


def _xi(g):
    """The grid's pixel centres, float32 like the framework's."""
    w, h = g.nx * g.ss, g.ny * g.ss
    step = np.float64(np.float32(g.pix) / np.float32(g.ss))
    x = (np.float64(g.cx) + (np.arange(w) - 0.5 * (w - 1)) * step).astype(np.float32)
    y = (np.float64(g.cy) + (np.arange(h) - 0.5 * (h - 1)) * step).astype(np.float32)
    return np.stack([np.broadcast_to(x, (h, w)), np.broadcast_to(y[:, None], (h, w))], -1).reshape(-1, 2)


def _arc_image(rng, c, lens, scale):
    """Observed pixels: a bright ring about the lens, and noise."""
    p = _xi(Grid(c["nx"], c["ny"], 1, c["pix"])).astype(np.float64)
    r = np.hypot(p[:, 0] - lens.x0, p[:, 1] - lens.y0)
    ring = np.exp(-0.5 * ((r - lens.theta_e) / (0.25 * lens.theta_e)) ** 2) * (1.5 + p[:, 0] / (r + 0.1))
    return (scale * ring + 0.1 * scale * rng.standard_normal(len(p))).astype(np.float32)


def _train_sources(c, g):
    """(inducing grid or None, length scale) of a training step."""
    if c["source"] == "self":
        return None, c["ell"]
    if c["src_pix"]:
        return Grid(c["side"], c["side"], 1, c["src_pix"]), c["ell"]
    yg = inducing_grid(g, c["side"])
    return yg, float(np.float32(yg.pix * 4.0 / 3.0))  # the paper's ratio of 40 mas to 30 mas


def _mhi(c):
    return (1e6 if c.get("n_sub", 0) >= 1000 else 1e7), 1e10


def _sides(c):
    """Image sides of a serving batch, from the largest down, even in their logarithm."""
    lo, hi, r = c["side_lo"], c["side_hi"], c["requests"]
    return [int(round(hi * (lo / hi) ** (k / max(r - 1, 1)))) for k in range(r)]


def _host_inputs(c, seed):
    """The case's inputs as host arrays and plain structs."""
    rng = _rng(c, seed)
    kind = c["kind"]
    if kind == "serve":
        reqs = []
        for k, side in enumerate(_sides(c)):
            cc = dict(nx=side, ny=side, pix=0.05)
            g, lens = Grid(side, side, 2, 0.05), _lens(rng, cc)
            sub = draw_subhalos(rng, c["max_sub"] * (k + 1) // c["requests"], lens, 1e7, 1e10)
            yg = inducing_grid(g, 128)
            p = Problem("request", g, lens, sub, 0, yg, float(np.float32(yg.pix * 4.0 / 3.0)), 1.0,
                        draw_v(rng, yg.n), 0)
            reqs.append((p, rng.standard_normal(p.n, dtype=np.float32)))
        return dict(reqs=reqs, step=1e-3)
    g, lens = _grid(c), _lens(rng, c)
    h = dict(g=g, lens=lens, sub=draw_subhalos(rng, c.get("n_sub", 0), lens, *_mhi(c)))
    if kind == "train":
        h["yg"], h["ell"] = _train_sources(c, g)
        h["v"] = draw_v(rng, h["yg"].n if h["yg"] else g.n)
        h["scale"] = 4.0 if h["yg"] else 20.0
        h["data"], h["noise"] = _arc_image(rng, c, lens, h["scale"]), 0.1 * h["scale"]
        h["variance"] = 1.0
    elif kind == "predict":
        h["yg"] = inducing_grid(g, c["side"])
        h["ell"], h["v"] = float(np.float32(h["yg"].pix * 4.0 / 3.0)), draw_v(rng, h["yg"].n)
    elif kind == "reconstruct":
        h["out_grid"], h["ell"] = Grid(c["out"], c["out"], 1, c["fov"] / c["out"]), c["ell"]
        h["v"] = rng.standard_normal((g.n, c["nrhs"]), dtype=np.float32)
    elif kind == "layers":
        h["yg"] = inducing_grid(g, c["side"])
        e = h["yg"].pix * 4.0 / 3.0
        h["ells"] = [float(np.float32(e * r)) for r in (1.0, 0.447, 0.2)[: c["layers"]]]
        h["vars"] = [1.0, 0.5, 0.25][: c["layers"]]
        shape = (c["layers"], h["yg"].n) + ((c["nrhs"],) if c["nrhs"] > 1 else ())
        h["v"] = rng.standard_normal(shape, dtype=np.float32)
    elif kind == "raytrace":
        xi = _xi(g)
        r = np.hypot(xi[:, 0], xi[:, 1])
        h["xi"] = xi[(r >= c["r_in"]) & (r <= c["r_out"])]
        # dL/dbeta of a smooth residual with noise
        n = len(h["xi"])
        h["d_beta"] = (np.cos(1.3 * h["xi"] + 0.4) + 0.3 * rng.standard_normal((n, 2))).astype(np.float32)
    elif kind == "windowed":
        h["v"] = rng.standard_normal(g.n, dtype=np.float32) * np.float32(c["ell"] ** 2)
        h["gout"] = (_arc_image(rng, c, lens, 1.0)).astype(np.float32)
    elif kind == "svi":
        m = c["side"] ** 2
        theta = np.array([lens.x0, lens.y0, lens.q, lens.phi, lens.theta_e, lens.g1, lens.g2])
        h["guide"] = dict(
            mu=np.concatenate([theta, 0.5 * rng.standard_normal(m)]), L=np.diag(np.full(7, 1e-3)),
            C=1e-3 * rng.standard_normal((m, 7)), sd_sp=np.full(m, 0.05),
            mu_layers=[0.3 * rng.standard_normal(g.n) for _ in range(c["layers"])],
            sd_layers=[np.full(g.n, 0.02) for _ in range(c["layers"])])
        f32 = lambda a: np.asarray(a, np.float32)  # noqa: E731
        h["guide"] = {k: [f32(x) for x in v] if isinstance(v, list) else f32(v) for k, v in h["guide"].items()}
        h["data"] = _arc_image(rng, c, lens, 2.0)
        h["eps_sp"] = rng.standard_normal(7 + m, dtype=np.float32)
        h["eps_layers"] = [rng.standard_normal(g.n, dtype=np.float32) for _ in range(c["layers"])]
    return h


def _sources_xy(h):
    """The ray-traced pixels of an earlier step, as a program holds them (float32)."""
    return _trace64(_xi(h["g"]), h["lens"], h["sub"]).float().contiguous()


class _Server:
    """The serving handle a program keeps open; closed with the state."""

    def __init__(self):
        self.session = Session(max_slots=16)

    def __del__(self):
        self.session.close()


def prepare(case, seed):
    c, h = dict(case), _host_inputs(case, seed)
    kind = c["kind"]
    s = dict(case=c, h=h)
    if kind == "serve":
        s["server"] = _Server()
        return s
    s["sub"] = _dev(h["sub"]) if len(h["sub"]) else None
    if kind == "train":
        leaf = lambda a: torch.tensor(a, dtype=torch.float32, device="cuda", requires_grad=True)  # noqa: E731
        s.update(v=_dev(h["v"]).requires_grad_(), lens=leaf(list(h["lens"].astuple())), ell=leaf(h["ell"]),
                 variance=leaf(h["variance"]), data=_dev(h["data"]))
        if s["sub"] is not None:
            s["sub"].requires_grad_()
    elif kind in ("predict", "layers"):
        s["v"] = _dev(h["v"])
    elif kind == "reconstruct":
        s.update(xy=_sources_xy(h), v=_dev(h["v"]) if c["nrhs"] > 1 else _dev(h["v"][:, 0]))
    elif kind == "raytrace":
        s.update(xi=_dev(h["xi"]), d_beta=_dev(h["d_beta"]))
    elif kind == "windowed":
        s.update(p=_sources_xy(h), v=_dev(h["v"]), gout=_dev(h["gout"]))
    elif kind == "density":
        s["p"] = _sources_xy(h)
    elif kind == "svi":
        gd = {k: [_dev(x) for x in v] if isinstance(v, list) else _dev(v) for k, v in h["guide"].items()}
        s.update(guide=svi.Guide(**gd), data=_dev(h["data"]), eps_sp=_dev(h["eps_sp"]),
                 eps_layers=[_dev(e) for e in h["eps_layers"]])
        s["cfg"] = _svi_config(c, h)
    return s


def _svi_config(c, h):
    return svi.ModelConfig(pixels=h["g"], source_grid=Grid(c["side"], c["side"], 1, c["src_pix"]),
                           sigma_sp=c["sigma_sp"], sigma_layers=list(SIGMA_LAYERS[: c["layers"]]), alpha_sp=1.934656,
                           alpha_layers=list(ALPHA_LAYERS[: c["layers"]]), noise=0.1, gamma=h["lens"].gamma)


# ---------------------------------------------------------------- one pass
def run(s):
    c, h = s["case"], s["h"]
    kind = c["kind"]
    if kind == "train":
        leaves = [s["v"], s["lens"], s["ell"], s["variance"]] + ([s["sub"]] if s["sub"] is not None else [])
        for t in leaves:
            t.grad = None
        f = lensed_gp_matvec(s["v"], s["lens"], s["sub"], s["ell"], s["variance"], h["g"], h["yg"])
        nll, g, _ = api.gaussian_nll(f.detach(), s["data"], h["noise"], grid=h["g"])
        f.backward(g)
        return {"loss": nll.float(), "f": f.detach(), "grads": [t.grad for t in leaves]}
    if kind == "predict":
        q = api.Points(grid=h["g"], lens=h["lens"], sub=s["sub"])
        f, beta = api.gp_kernel_matvec(q, api.Points(grid=h["yg"]), s["v"], h["ell"], 1.0, want_beta=True)
        return {"f": f, "beta": beta}
    if kind == "reconstruct":
        src = api.Points(xy=s["xy"], grid=h["g"])  # the pixels in their image layout
        return api.gp_kernel_matvec(api.Points(grid=h["out_grid"]), src, s["v"], h["ell"], 1.0)
    if kind == "layers":
        q = api.Points(grid=h["g"], lens=h["lens"], sub=s["sub"])
        return api.gp_kernel_matvec_layers(q, api.Points(grid=h["yg"]), s["v"], h["ells"], h["vars"])
    if kind == "raytrace":
        pts = api.Points(xy=s["xi"], lens=h["lens"], sub=s["sub"])
        beta, alpha = api.lens_raytrace(pts, want_alpha=True)
        d_lens, d_sub = api.lens_raytrace_vjp(pts, s["d_beta"])
        return {"beta": beta, "alpha": alpha, "d_lens": d_lens.float(), "d_sub": d_sub.float()}
    if kind == "windowed":
        p, g = s["p"], h["g"]
        z = api.pixel_shapes(p, g.nx, g.ny)
        me = api.Points(xy=p, grid=g)
        f = api.gp_windowed_matvec(p, z, me, s["v"], c["ell"], layout=g)
        G = api.gp_windowed_matvec_bwd(p, z, me, s["v"], c["ell"], s["gout"], want=("v", "p", "q", "z"), layout=g)
        return {"shapes": z, "f": f, "d": G, "p_of_z": api.pixel_shapes_vjp(p, g.nx, g.ny, G["z"])}
    if kind == "density":
        r2, a = api.knn_density(s["p"], c["k"], lengthscale=c["ell"])
        return {"r2": r2, "A": a}
    if kind == "svi":
        loss, G = svi.loss_and_grads(s["cfg"], s["guide"], s["data"], s["eps_sp"], s["eps_layers"])
        return {"loss": loss.float(), **{k: G[k] for k in ("mu", "L", "C", "sd_sp", "layers_mu", "layers_sd")}}
    S = s["server"].session
    tickets = [S.submit(p, d, c["iters"], h["step"]) for p, d in h["reqs"]]
    res = [S.poll(t, timeout_s=300) for t in tickets]
    assert all(r.status == 0 for r in res), [r.status for r in res]
    return [{"f": r.out, "v": r.v, "d_lens": r.d_lens.astype(np.float32), "d_sub": r.d_sub.astype(np.float32),
             "loss": np.float32(r.loss)} for r in res]


# ---------------------------------------------------------------- what a pass cannot do without
def _near(ell, density, m):
    """Sources whose kernel value is not zero in float32: exp(-d^2 / (2 l^2)) >= 2^-126."""
    return min(m, math.pi * 2.0 * 126.0 * math.log(2.0) * ell * ell * density)


def work(case):
    """bytes: each input read and each output written once. flops: per kernel pair
    whose value is not zero (counted at the image's own density of points, no
    magnification), 8 to form the pair's value and 2 per sum it enters; per
    point and subhalo 12, a far-field deflection; per point 300 for the lens."""
    c = case
    kind = c["kind"]
    if kind == "serve":
        n = 4 * sum(side * side for side in _sides(c))
        pairs = n * _near(4 / 3, 1.0, 16384)
        one = pairs * (8 + 2 * 4 + 8 + 2) + n * (300 + 600) + n * 0.4 * c["max_sub"] * 36
        return {"bytes": n * 8 + c["requests"] * 16384 * 8, "flops": c["iters"] * one}
    n = c["nx"] * c["ny"] * c.get("ss", 1) ** 2
    dens = (c.get("ss", 1) / c["pix"]) ** 2
    S = c.get("n_sub", 0)
    trace = n * (300 + 12 * S)
    if kind == "train":
        if c["source"] == "self":
            m, near, vb = n, _near(c["ell"], dens, n), 4 * n
        else:
            m = c["side"] ** 2
            near = _near(c["ell"] / c["src_pix"], 1.0, m) if c["src_pix"] else _near(4 / 3, 1.0, m)
            vb = 4 * m
        return {"bytes": 2 * vb + 4 * n + 4 * c["nx"] * c["ny"] + 40 * S, "flops":
                n * near * (8 + 2 + 8 + 2 * 7) + trace * 3}
    if kind == "predict":
        return {"bytes": 4 * c["side"] ** 2 + 12 * n + 20 * S,
                "flops": n * _near(4 / 3, 1.0, c["side"] ** 2) * 10 + trace}
    if kind == "reconstruct":
        q = c["out"] ** 2
        return {"bytes": n * (8 + 4 * c["nrhs"]) + 4 * q * c["nrhs"],
                "flops": q * _near(c["ell"], dens, n) * (8 + 2 * c["nrhs"])}
    if kind == "layers":
        m = c["side"] ** 2
        near = sum(_near(4 / 3 * r, 1.0, m) for r in (1.0, 0.447, 0.2)[: c["layers"]])
        return {"bytes": 4 * c["layers"] * m * c["nrhs"] + 4 * n * c["nrhs"] + 20 * S,
                "flops": n * near * (4 + 2 * c["nrhs"]) + trace}
    if kind == "raytrace":
        frac = min(1.0, math.pi * (c["r_out"] ** 2 - c["r_in"] ** 2) / (c["nx"] * c["ny"] * c["pix"] ** 2))
        return {"bytes": frac * n * 32 + S * 36, "flops": 3 * frac * trace}
    if kind in ("windowed", "svi"):
        # windows about the size of a pixel: C = Z + l^2 / 2, Z ~ pix^2 / (4 pi)
        ells = [c["ell"]] if kind == "windowed" else SIGMA_LAYERS[: c["layers"]]
        near = sum(_near(math.sqrt(c["pix"] ** 2 / (4 * math.pi) + 0.5 * e * e), dens, n) for e in ells)
        b, f = (4 * n * len(ells)) * 5, n * near * (14 + 2 + 14 + 2 * 9) + 300 * n
        if kind == "svi":
            m = c["side"] ** 2
            f += n * _near(c["sigma_sp"] / math.sqrt(2.0) / c["src_pix"], 1.0, m) * 32 + 3 * trace
            return {"bytes": b + 4 * n + 4 * m * 20, "flops": f}
        return {"bytes": b + n * (8 + 12 + 4 + 16 + 12 + 8), "flops": f}
    return {"bytes": n * 16, "flops": n * c["k"] * 12}


# ---------------------------------------------------------------- the same in 64 bits, in plain torch
def _f64(a):
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    t = torch.from_numpy(np.ascontiguousarray(a)) if isinstance(a, np.ndarray) else torch.as_tensor(a)
    return t.to(dev, torch.float64)


def _sple64(x, y, L, gamma):
    """Deflection of the singular power-law ellipsoid and the shear."""
    x0, y0, q, phi, te, g1, g2 = L
    co, si = torch.cos(phi), torch.sin(phi)
    u, v = co * (x - x0) + si * (y - y0), co * (y - y0) - si * (x - x0)
    X, Y = torch.sqrt(q) * u, v / torch.sqrt(q)
    r2 = X * X + Y * Y  # the centre itself deflects nothing
    R = torch.sqrt(torch.where(r2 > 0, r2, torch.ones_like(r2)))
    ex, ey = X / R, Y / R
    f = (1 - q) / (1 + q)
    zr, zi = -f * (ex * ex - ey * ey), -f * 2 * ex * ey
    a, b = 0.5 * (gamma - 1.0), 0.5 * (5.0 - gamma)
    tr, ti = torch.ones_like(R), torch.zeros_like(R)
    Fr, Fi = tr, ti
    for k in range(1, 2 + int(math.ceil(-39.0 / math.log(max(float(f.detach()), 1e-8))))):
        w = (a + k - 1.0) / (b + k - 1.0)
        tr, ti = w * (tr * zr - ti * zi), w * (tr * zi + ti * zr)
        Fr, Fi = Fr + tr, Fi + ti
    pre = te * 2 * torch.sqrt(q) / (1 + q) * (te / R) ** (gamma - 2.0)
    pre = torch.where(r2 > 0, pre, torch.zeros_like(pre))
    ar, ai = pre * (Fr * ex - Fi * ey), pre * (Fr * ey + Fi * ex)
    return co * ar - si * ai + g1 * x + g2 * y, si * ar + co * ai + g2 * x - g1 * y


def _tnfw64(x, y, sub):
    """Summed deflection of truncated-NFW subhalos (Baltz, Marshall & Oguri 2009)."""
    dx, dy = x[:, None] - sub[:, 0], y[:, None] - sub[:, 1]
    ks, ts, tau = sub[:, 2], sub[:, 3], sub[:, 4]
    x2 = (dx * dx + dy * dy) / (ts * ts)
    e = x2 - 1.0
    near = e.abs() < 1e-4
    out = torch.where(near | (e < 0), torch.ones_like(e), e)
    ins = torch.where(near | (e > 0), torch.full_like(e, -0.5), e)
    so, si = torch.sqrt(out), torch.sqrt(-ins)
    F = torch.where(e > 0, torch.atan(so) / so, torch.atanh(si) / si)
    F = torch.where(near, 1 - e * (1 / 3 - e * (1 / 5 - e / 7)), F)
    t2 = tau * tau
    st = torch.sqrt(t2 + x2)
    lx = 0.5 * torch.log(x2) - torch.log(st + tau)
    B = (t2 + 1 + 2 * e) * F + tau * math.pi + (t2 - 1) * torch.log(tau) + st * ((t2 - 1) / tau * lx - math.pi)
    m = 4 * ks * t2 / ((t2 + 1) * (t2 + 1)) * B / x2
    return (m * dx).sum(1), (m * dy).sum(1)


def _blocks(n, per):
    return [slice(i, min(i + per, n)) for i in range(0, n, per)]


def _alpha64(xi, L, gamma, sub):
    ax, ay = _sple64(xi[:, 0], xi[:, 1], L, gamma)
    if sub is not None and len(sub):
        bx, by = _tnfw64(xi[:, 0], xi[:, 1], sub)
        ax, ay = ax + bx, ay + by
    return torch.stack([ax, ay], 1)


def _lens7(lens):
    p = lens.astuple()
    return _f64([p[0], p[1], p[2], p[3], p[4], p[6], p[7]])


def _trace64(xi, lens, sub, alpha=False):
    xi, L, sub = _f64(xi), _lens7(lens), _f64(sub)
    per = max(1, 20_000_000 // max(len(sub), 30))
    with torch.no_grad():
        a = torch.cat([_alpha64(xi[b], L, lens.gamma, sub) for b in _blocks(len(xi), per)])
    return (xi - a, a) if alpha else xi - a


def _trace_grad64(xi, lens, sub, d_beta):
    """(d_lens[7], d_sub[S, 4])."""
    xi = _f64(xi)
    L, sub = _lens7(lens).requires_grad_(), _f64(sub).requires_grad_()
    for b in _blocks(len(xi), max(1, 8_000_000 // max(len(sub), 30))):
        (_alpha64(xi[b], L, lens.gamma, sub) * -d_beta[b]).sum().backward()
    ds = sub.grad[:, :4] if sub.grad is not None else torch.zeros((0, 4), dtype=torch.float64, device=xi.device)
    return L.grad, ds


def _row_blocks(n, grid, side=64):
    """Index lists of the rows: tiles of the image where there is one."""
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    if grid is None:
        return [torch.arange(b.start, b.stop, device=dev) for b in _blocks(n, side * side)]
    w, h = grid.nx * grid.ss, grid.ny * grid.ss
    i = torch.arange(n, device=dev).reshape(h, w)
    return [i[r:r + side, k:k + side].reshape(-1) for r in range(0, h, side) for k in range(0, w, side)]


def _reach(x, y, r):
    """Sources within r of the box of the points x: the others are below 1e-26 of a pair at distance 0."""
    lo, hi = x.min(0).values, x.max(0).values
    d = torch.clamp(torch.maximum(lo - y, y - hi), min=0.0)
    return torch.nonzero((d * d).sum(1) <= r * r).squeeze(1)


_CUT = math.sqrt(120.0)  # exp(-60)


def _reduce64(x, y, v, ell, var, rows):
    """sum_j var exp(-|x_i - y_j|^2 / 2 l^2) v_j; v (m, r)."""
    ell = float(np.float32(ell))
    out = torch.zeros((len(x), v.shape[1]), dtype=torch.float64, device=x.device)
    for i in rows:
        j = _reach(x[i], y, _CUT * ell)
        if len(j):
            for b in _blocks(len(i), max(1, 60_000_000 // len(j))):
                a, yb = x[i[b]], y[j]
                d2 = (a[:, 0, None] - yb[:, 0]) ** 2 + (a[:, 1, None] - yb[:, 1]) ** 2
                out[i[b]] = var * (torch.exp(d2 * (-0.5 / ell ** 2)) @ v[j])
    return out


def _reduce_grad64(x, y, v, ell, var, g, rows, self_=False):
    """(d_v, d_x, d_len, d_var) of sum_i g_i out_i, one right-hand side."""
    ell = float(np.float32(ell))
    dv = torch.zeros_like(v)
    dx, dy = torch.zeros_like(x), torch.zeros_like(y)
    dl = dvar = 0.0
    for i in rows:
        j = _reach(x[i], y, _CUT * ell)
        if not len(j):
            continue
        for b in _blocks(len(i), max(1, 60_000_000 // len(j))):
            ib = i[b]
            a, yb = x[ib], y[j]
            ex, ey = yb[:, 0] - a[:, 0, None], yb[:, 1] - a[:, 1, None]
            d2 = ex * ex + ey * ey
            K = var * torch.exp(d2 * (-0.5 / ell ** 2))
            dv.index_add_(0, j, g[ib] @ K)
            K *= g[ib][:, None] * v[j]
            dvar += K.sum() / var
            dl += (K * d2).sum() / ell ** 3
            ex *= K / ell ** 2
            ey *= K / ell ** 2
            dx[ib] = torch.stack([ex.sum(1), ey.sum(1)], 1)
            if self_:
                dy.index_add_(0, j, -torch.stack([ex.sum(0), ey.sum(0)], 1))
    return dv, dx + dy if self_ else dx, dl, dvar


def _shapes64(p, W, H):
    P = p.reshape(H, W, 2)
    ax = torch.cat([P[:, 1:2] - P[:, :1], 0.5 * (P[:, 2:] - P[:, :-2]), P[:, -1:] - P[:, -2:-1]], 1)
    by = torch.cat([P[1:2] - P[:1], 0.5 * (P[2:] - P[:-2]), P[-1:] - P[-2:-1]], 0)
    z = [ax[..., a] * ax[..., b] + by[..., a] * by[..., b] for a, b in ((0, 0), (0, 1), (1, 1))]
    return torch.stack(z, -1).reshape(-1, 3) / (4 * math.pi)


def _windowed64(p, z, v, ell, g, rows):
    """The image-plane layer's reduction and, with g, its gradients (d_v, d_p, d_q, d_z)."""
    ell = float(np.float32(ell))
    c = z + _f64([0.5 * ell ** 2, 0.0, 0.5 * ell ** 2])
    det = c[:, 0] * c[:, 2] - c[:, 1] ** 2
    M = torch.stack([c[:, 2], -c[:, 1], c[:, 0]], 1) / det[:, None]
    norm = 1.0 / (2 * math.pi * torch.sqrt(det))
    lmax = 0.5 * (c[:, 0] + c[:, 2]) + torch.sqrt(0.25 * (c[:, 0] - c[:, 2]) ** 2 + c[:, 1] ** 2)
    f, dv, dp, dq, dz = torch.zeros_like(v), torch.zeros_like(v), torch.zeros_like(p), torch.zeros_like(p), \
        torch.zeros_like(z)
    order = [i[torch.argsort(lmax[i])] for i in rows]  # the few wide windows of a tile by themselves
    for ib in [o[b] for o in order for b in _blocks(len(o), 256)]:
        j = _reach(p[ib], p, _CUT * math.sqrt(float(lmax[ib].max())))
        a, q, m = p[ib], p[j], M[ib]
        ex, ey = a[:, 0, None] - q[:, 0], a[:, 1, None] - q[:, 1]
        ux = m[:, 0, None] * ex + m[:, 1, None] * ey
        uy = m[:, 1, None] * ex + m[:, 2, None] * ey
        G = norm[ib][:, None] * torch.exp(-0.5 * (ex * ux + ey * uy))
        f[ib] = G @ v[j]
        if g is None:
            continue
        G *= g[ib][:, None]
        dv.index_add_(0, j, G.sum(0))
        G *= v[j]
        s0 = G.sum(1)
        gx, gy = G * ux, G * uy
        dp[ib] = -torch.stack([gx.sum(1), gy.sum(1)], 1)
        dq.index_add_(0, j, torch.stack([gx.sum(0), gy.sum(0)], 1))
        dz[ib] = torch.stack([0.5 * ((gx * ux).sum(1) - m[:, 0] * s0), (gx * uy).sum(1) - m[:, 1] * s0,
                              0.5 * ((gy * uy).sum(1) - m[:, 2] * s0)], 1)
    return f, dv, dp, dq, dz


def _knn64(p, k):
    """Squared distance to the k-th nearest other point: strips of the points
    sorted by x, each against the points within its own bound on the distance."""
    order = torch.argsort(p[:, 0])
    s = p[order].contiguous()
    xs = s[:, 0].contiguous()
    r2 = torch.empty(len(p), dtype=torch.float64, device=p.device)
    kk = min(k + 1, len(p))
    for b in _blocks(len(p), 4096):
        a = s[b]
        wide = s[max(0, b.start - 512):b.stop + 512]
        d = (a[:, 0, None] - wide[:, 0]) ** 2 + (a[:, 1, None] - wide[:, 1]) ** 2
        r = torch.sqrt(torch.topk(d, kk, dim=1, largest=False).values[:, -1])
        for h in torch.argsort(r).split(512):  # points of like bounds together
            lo = int(torch.searchsorted(xs, (a[h, 0] - r[h]).min()))
            hi = int(torch.searchsorted(xs, (a[h, 0] + r[h]).max(), right=True))
            d = (a[h, 0, None] - s[lo:hi, 0]) ** 2 + (a[h, 1, None] - s[lo:hi, 1]) ** 2
            r2[order[b][h]] = torch.topk(d, kk, dim=1, largest=False).values[:, -1]
    return r2


def _svi64(c, h):
    L2PI = math.log(2 * math.pi)
    cfg, gd = _svi_config(c, h), {k: [_f64(x) for x in v] if isinstance(v, list) else _f64(v)
                                  for k, v in h["guide"].items()}
    g, eps, m = h["g"], _f64(h["eps_sp"]), c["side"] ** 2
    L = torch.tril(gd["L"])
    theta = gd["mu"][:7] + L @ eps[:7]
    y_sp = gd["mu"][7:] + gd["C"] @ eps[:7] + gd["sd_sp"] * eps[7:]
    logq = -0.5 * (eps @ eps) - torch.log(torch.diag(L)).sum() - torch.log(gd["sd_sp"]).sum() - 0.5 * (7 + m) * L2PI
    th = theta.clone().requires_grad_()
    xi = _f64(_xi(g))
    beta_g = xi - _alpha64(xi, [th[k] for k in range(7)], cfg.gamma, None)
    beta = beta_g.detach()
    sg = cfg.source_grid
    s_sp = cfg.sigma_sp
    a_sp = math.sqrt(2 * math.pi) * s_sp * sg.pix / (math.pi * s_sp ** 2)
    yg, ell = _f64(_xi(sg)), s_sp / math.sqrt(2.0)
    rows = _row_blocks(g.n, g)
    w_sp = (a_sp * y_sp)
    f = _reduce64(beta, yg, w_sp[:, None], ell, 1.0, rows)[:, 0]
    z = _shapes64(beta, g.nx, g.ny)
    r2 = _knn64(beta, cfg.knn_k)
    terms, ws, As = 0.0, [], []
    for mu, sd, e, al, s in zip(gd["mu_layers"], gd["sd_layers"], h["eps_layers"], cfg.alpha_layers,
                                cfg.sigma_layers):
        e = _f64(e)
        y = mu + sd * e
        A = math.pi * s * torch.sqrt(2 * r2 / cfg.knn_k)
        f = f + _windowed64(beta, z, A * y, s, None, rows)[0]
        terms = terms + (y * y).sum() / (2 * al * al) + g.n * (math.log(al) + 0.5 * L2PI) \
            - (0.5 * e * e + torch.log(sd)).sum() - 0.5 * g.n * L2PI
        ws.append((y, A))
    d = _f64(h["data"])
    res = f - d
    al = cfg.alpha_sp
    loss = (0.5 * res * res).sum() / cfg.noise ** 2 + g.n * (math.log(cfg.noise) + 0.5 * L2PI) + logq + terms \
        + (y_sp * y_sp).sum() / (2 * al * al) + m * (math.log(al) + 0.5 * L2PI)
    gf = res / cfg.noise ** 2
    d_beta, d_z = torch.zeros_like(beta), torch.zeros_like(z)
    l_mu, l_sd = [], []
    for (y, A), sd, e, al_l, s in zip(ws, gd["sd_layers"], h["eps_layers"], cfg.alpha_layers, cfg.sigma_layers):
        _, dv, dp, dq, dz = _windowed64(beta, z, A * y, s, gf, rows)
        d_beta, d_z = d_beta + dp + dq, d_z + dz
        t = A * dv + y / al_l ** 2
        l_mu.append(t)
        l_sd.append(t * _f64(e) - 1.0 / sd)
    b = beta.clone().requires_grad_()
    (_shapes64(b, g.nx, g.ny) * d_z).sum().backward()
    dv, dx, _, _ = _reduce_grad64(beta, yg, w_sp, ell, 1.0, gf, rows)
    beta_g.backward(d_beta + b.grad + dx)
    d_x = torch.cat([th.grad, a_sp * dv + y_sp / al ** 2])
    d_L = torch.tril(torch.outer(d_x[:7], eps[:7])) - torch.diag(1.0 / torch.diag(L))
    return {"loss": loss, "mu": d_x, "L": d_L, "C": torch.outer(d_x[7:], eps[:7]),
            "sd_sp": d_x[7:] * eps[7:] - 1.0 / gd["sd_sp"], "layers_mu": l_mu, "layers_sd": l_sd}


def _chain64(h, v, g_of):
    """Forward and backward of one lens system: (f, loss, d_v, d_len, d_var, d_lens7, d_sub)."""
    xi = _xi(h["g"])
    beta = _trace64(xi, h["lens"], h["sub"])
    y = beta if h["yg"] is None else _f64(_xi(h["yg"]))
    rows = _row_blocks(h["g"].n, h["g"])
    ell, var = h["ell"], h["variance"]
    f = _reduce64(beta, y, v[:, None], ell, var, rows)[:, 0]
    loss, g = g_of(f)
    dv, dx, dl, dvar = _reduce_grad64(beta, y, v, ell, var, g, rows, h["yg"] is None)
    return (f, loss, dv, dl, dvar) + _trace_grad64(xi, h["lens"], h["sub"], dx)


def exact(case, seed):
    c, h = dict(case), _host_inputs(case, seed)
    kind = c["kind"]
    if kind == "train":
        g, s = h["g"], h["noise"]

        def nll(f):
            img = f.reshape(g.ny, g.ss, g.nx, g.ss).mean((1, 3)).reshape(-1)
            r = img - _f64(h["data"])
            up = (r / (s * s * g.ss ** 2)).reshape(g.ny, 1, g.nx, 1).expand(g.ny, g.ss, g.nx, g.ss)
            loss = 0.5 * (r * r).sum() / s ** 2 + len(r) * (math.log(s) + 0.5 * math.log(2 * math.pi))
            return loss, up.reshape(-1)

        f, loss, dv, dl, dvar, d7, ds = _chain64(h, _f64(h["v"]), nll)
        d8 = torch.cat([d7[:5], d7.new_zeros(1), d7[5:]])  # the slope is held fixed
        grads = [dv, d8, dl.reshape(()), dvar.reshape(())]
        return {"loss": loss, "f": f, "grads": grads + ([torch.cat([ds, ds.new_zeros(len(ds), 1)], 1)]
                                                        if len(ds) else [])}
    if kind == "predict":
        beta = _trace64(_xi(h["g"]), h["lens"], h["sub"])
        f = _reduce64(beta, _f64(_xi(h["yg"])), _f64(h["v"])[:, None], h["ell"], 1.0, _row_blocks(h["g"].n, h["g"]))
        return {"f": f[:, 0], "beta": beta}
    if kind == "reconstruct":
        x, v = _f64(_xi(h["out_grid"])), _f64(h["v"])
        f = _reduce64(x, _sources_xy(h).double(), v, h["ell"], 1.0, _row_blocks(len(x), h["out_grid"]))
        return f if c["nrhs"] > 1 else f[:, 0]
    if kind == "layers":
        beta, y, v = _trace64(_xi(h["g"]), h["lens"], h["sub"]), _f64(_xi(h["yg"])), _f64(h["v"])
        rows = _row_blocks(len(beta), h["g"])
        f = sum(_reduce64(beta, y, v[k].reshape(len(y), -1), e, w, rows)
                for k, (e, w) in enumerate(zip(h["ells"], h["vars"])))
        return f if c["nrhs"] > 1 else f[:, 0]
    if kind == "raytrace":
        beta, alpha = _trace64(h["xi"], h["lens"], h["sub"], alpha=True)
        d7, ds = _trace_grad64(h["xi"], h["lens"], h["sub"], _f64(h["d_beta"]))
        return {"beta": beta, "alpha": alpha, "d_lens": d7, "d_sub": ds}
    if kind == "windowed":
        p, g = _sources_xy(h).double(), h["g"]
        b = p.clone().requires_grad_()
        z = _shapes64(b, g.nx, g.ny)
        f, dv, dp, dq, dz = _windowed64(p, z.detach(), _f64(h["v"]), c["ell"], _f64(h["gout"]), _row_blocks(g.n, g))
        z.backward(dz)
        return {"shapes": z.detach(), "f": f, "d": {"v": dv, "p": dp, "q": dq, "z": dz}, "p_of_z": b.grad}
    if kind == "density":
        r2 = _knn64(_sources_xy(h).double(), c["k"])
        return {"r2": r2, "A": math.pi * c["ell"] * torch.sqrt(2 * r2 / c["k"])}
    if kind == "svi":
        return _svi64(c, h)
    out = []
    for p, data in h["reqs"]:
        hh = dict(g=p.xgrid, lens=p.lens, sub=p.sub, yg=p.ygrid, ell=p.lengthscale, variance=p.variance)
        beta, y, v = _trace64(_xi(hh["g"]), hh["lens"], hh["sub"]), _f64(_xi(hh["yg"])), _f64(p.v)
        rows, d = _row_blocks(p.n, p.xgrid), _f64(data)
        for k in range(c["iters"]):
            f = _reduce64(beta, y, v[:, None], p.lengthscale, p.variance, rows)[:, 0]
            dv, dx, _, _ = _reduce_grad64(beta, y, v, p.lengthscale, p.variance, f - d, rows)
            v = v - float(np.float32(h["step"])) * dv
        d7, ds = _trace_grad64(_xi(hh["g"]), hh["lens"], hh["sub"], dx)
        out.append({"f": f, "v": v, "d_lens": d7, "d_sub": ds, "loss": 0.5 * ((f - d) ** 2).sum()})
    return out
