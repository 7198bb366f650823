"""The calls whose speed matters to a program that uses this framework.

Each case is one evaluation through the public Python entry points, with the
inputs of ``workloads.py`` (the paper's lattice patches and Lamb-Oseen vortex,
uniform points, Gaussian clusters) drawn on the GPU.  ``prepare`` holds what a
simulation keeps between its time steps -- the context and the particles --
and ``run`` is one velocity (or potential) evaluation as a time step calls it.
"""
import math

import numpy as np
import torch

from paper_0905_2637_gb300 import _lib, fmm3d

ORDERS = (8, 12, 17)


def listed():
    return [
        # The smallest request a simulation or the server makes: 64 x 64 blobs, plain launches.
        _case("patch-4k", "lattice", side=64, p=17),
        # The accuracy configuration: 10,000 uniform blobs, every stage in FP64.
        _case("uniform-10k-fp64", "uniform", n=10_000, L=4, p=12, sigma=0.005, precision="fp64",
              dtype="f64"),
        # An ordinary vortex patch, 16 blobs per leaf, time steps replayed as a graph.
        _case("lattice-1M", "lattice", side=1024, L=8, p=17, graph=True),
        # The same patch as the FP64 reference solution that mixed runs are checked against.
        _case("lattice-1M-fp64", "lattice", side=1024, L=8, p=17, precision="fp64", dtype="f64"),
        # The paper's own experiment (875 x 875 blobs, one per occupied leaf).
        _case("lamb-oseen-765k", "lamb_oseen", half_width=7.0, L=10, p=17, sigma=0.02, graph=True),
        # The benchmark's headline workload, and the largest: strongly clustered blobs.
        _case("clustered-16M", "clustered", n=1 << 24, L=10, p=17, sigma=0.002, graph=True),
        # Clustered blobs in pinned host memory, copied in and out by the call itself.
        _case("clustered-4M-host", "clustered", n=1 << 22, L=9, p=17, sigma=0.004, graph=True,
              host=True),
        # Many independent uneven problems in one call, mixed orders, depth chosen by the library.
        _case("batch-512", "batch", count=512, n_min=1000, n_max=262_144, sizes=1, graph=True),
        # The second kernel, the logarithmic potential of a million charges.
        _case("laplace-1M", "laplace", n=1 << 20, L=8, p=17, graph=True),
        # Three dimensions: potential and field of two million uniform charges.
        _case("uniform3d-2M", "uniform3d", n=1 << 21, L=5, p=8),
        # Three dimensions, hot leaves beside empty ones.
        _case("clustered3d-2M", "clustered3d", n=1 << 21, L=6, p=8),
        # The 3D reference solution in FP64.
        _case("uniform3d-262k-fp64", "uniform3d", n=1 << 18, L=4, p=8, precision="fp64",
              dtype="f64"),
    ]


def _case(name, kind, **more):
    c = {"kind": kind, "precision": "mixed", "dtype": "f32", "graph": False, **more}
    if name:
        c["name"] = name
    if "L" not in c and kind != "batch":
        c["L"] = _depth(c)
    return c


def _depth(c):
    """The depth at the densities of the listed cases: 16 blobs (3D: 64 charges) per leaf."""
    if c["kind"].endswith("3d"):
        return max(2, round(math.log(c["n"] / 64, 8)))
    return max(2, round(math.log(_count(c) / 16, 4)))


def _count(c):
    if c["kind"] == "lattice":
        return c["side"] ** 2
    if c["kind"] == "lamb_oseen":
        return (2 * math.floor(c["half_width"] / (0.8 * c["sigma"])) + 1) ** 2
    if c["kind"] == "batch":
        return int(_batch_sizes(c)[0].sum())
    return c["n"]


def _log_int(rng, lo, hi):
    return int(math.exp(rng.uniform(math.log(lo), math.log(hi + 1))))


def draw(rng):
    kind = rng.choice(["lattice", "lattice", "clustered", "clustered", "uniform", "lamb_oseen",
                       "batch", "laplace", "uniform3d", "clustered3d"])
    graph = rng.random() < 0.5
    if kind == "batch":
        return _case(None, kind, count=_log_int(rng, 8, 256), n_min=1000,
                     n_max=_log_int(rng, 8000, 262_144), sizes=rng.randrange(1, 1000), graph=graph)
    fp64 = kind != "laplace" and rng.random() < 0.3
    more = dict(precision="fp64", dtype=rng.choice(["f64", "f64", "f32"])) if fp64 else {}
    if kind.endswith("3d"):
        top = 150_000 if fp64 else 1_500_000 if kind == "uniform3d" else 600_000
        return _case(None, kind, n=_log_int(rng, 5000, top), p=rng.randrange(4, 9), **more)
    more.update(p=rng.choice(ORDERS), graph=graph)
    if kind == "lattice":
        return _case(None, kind, side=_log_int(rng, 60, 900 if fp64 else 2000), **more)
    if kind == "clustered":
        return _case(None, kind, n=_log_int(rng, 20_000, 60_000 if fp64 else 4_000_000),
                     sigma=rng.choice([0.002, 0.004]), host=rng.random() < 0.25, **more)
    if kind == "lamb_oseen":
        return _case(None, kind, half_width=round(rng.uniform(1.0, 3.0 if fp64 else 8.0), 3),
                     sigma=0.02, **more)
    n = _log_int(rng, 4000, 400_000 if fp64 else 1_500_000)
    if kind == "uniform":
        return _case(None, kind, n=n, sigma=round(0.5 / math.sqrt(n), 6), **more)
    return _case(None, "laplace", n=n, **more)


# --------------------------------------------------------------------------- inputs

def _batch_sizes(c):
    """Sizes and orders of a batch: part of the case, so that every seed has the same ones."""
    r = np.random.default_rng(c["sizes"])
    n = np.floor(np.exp(r.uniform(math.log(c["n_min"]), math.log(c["n_max"]), c["count"])))
    return n.astype(np.int64), r.choice(np.array(ORDERS), c["count"])


def _uniform(g, *shape):
    return torch.rand(*shape, generator=g, device="cuda", dtype=torch.float64)


def _normal(g, *shape):
    return torch.randn(*shape, generator=g, device="cuda", dtype=torch.float64)


def _inputs(c, seed):
    """(coordinates, strengths, sigma, domain) in the case's storage type."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    dim = 3 if c["kind"].endswith("3d") else 2
    domain = (0.0,) * dim + (1.0,)
    sigma = c.get("sigma", 1.0)
    n = _count(c)
    if c["kind"] == "lattice":
        side = c["side"]
        h = 1.0 / side
        i = torch.arange(side, device="cuda", dtype=torch.float64)
        y, x = torch.meshgrid(i, i, indexing="ij")
        xs = [(v.reshape(-1) + 0.5 + 0.5 * (_uniform(g, n) - 0.5)) * h for v in (x, y)]
        q = h * h * torch.exp(-((xs[0] - 0.5) ** 2 + (xs[1] - 0.5) ** 2) / 0.01)
        sigma = 1.5 * h
    elif c["kind"] == "lamb_oseen":
        # the vortex strength and age differ by seed, the lattice is the paper's
        h = 0.8 * sigma
        m = math.floor(c["half_width"] / h)
        i = torch.arange(-m, m + 1, device="cuda", dtype=torch.float64) * h
        y, x = torch.meshgrid(i, i, indexing="ij")
        xs = [x.reshape(-1), y.reshape(-1)]
        four_nu_t = float(0.5 + torch.rand(1, generator=g, device="cuda"))
        q = torch.exp(-(xs[0] ** 2 + xs[1] ** 2) / four_nu_t) * (h * h / (math.pi * four_nu_t))
        edge = c["half_width"] + h
        domain = (-edge, -edge, 2 * edge)
    elif c["kind"] in ("clustered", "clustered3d"):
        centres = 0.2 + 0.6 * _uniform(g, 8, dim)
        std = 0.02 if dim == 2 else 0.04
        of = torch.randint(0, 8, (n,), generator=g, device="cuda")
        pts = (centres[of] + std * _normal(g, n, dim)).clamp_(0.0, 1.0)
        xs = [pts[:, k].contiguous() for k in range(dim)]
        q = _normal(g, n) / n
    else:
        xs = list(_uniform(g, dim, n))
        q = 2.0 * _uniform(g, n) - 1.0
        if dim == 3:
            q = q / n
    t = torch.float32 if c["dtype"] == "f32" else torch.float64
    return [v.to(t) for v in xs], q.to(t), sigma, domain


# --------------------------------------------------------------------------- the calls

def prepare(case, seed):
    c = case
    xs, q, sigma, domain = _inputs(c, seed)
    if c["kind"].endswith("3d"):
        ctx = fmm3d.Context3D(domain, c["L"], c["p"], precision=c["precision"], dtype=c["dtype"])
        return {"kind": "3d", "ctx": ctx, "args": (*xs, q)}
    if c["kind"] == "batch":
        ctx = _lib.Context((0, 0, 1), 2, 8, 0.01, precision=c["precision"], dtype=c["dtype"])
        u, v = torch.empty_like(q), torch.empty_like(q)
        sizes, orders = _batch_sizes(c)
        parts = [t.split(sizes.tolist()) for t in (*xs, q, u, v)]
        items = [dict(domain=domain, order=int(p), sigma=0.5 / math.sqrt(n), x=a[0], y=a[1],
                      gamma=a[2], u=a[3], v=a[4]) for n, p, *a in zip(sizes, orders, *parts)]
        state = {"kind": "batch", "ctx": ctx, "items": items, "out": {"u": u, "v": v}}
    else:
        ctx = _lib.Context(domain, c["L"], c["p"], sigma, precision=c["precision"],
                           dtype=c["dtype"],
                           kernel="laplace" if c["kind"] == "laplace" else "vortex")
        state = {"kind": "2d", "ctx": ctx, "args": (*xs, q)}
        if c.get("host"):
            host = [t.cpu().pin_memory() for t in (*xs, q)]
            out = [torch.empty_like(q, device="cpu").pin_memory() for _ in range(2)]
            state = {"kind": "host", "ctx": ctx, "args": host, "out": {"u": out[0], "v": out[1]}}
    if c["graph"]:
        ctx.set_option(_lib.PETFMM_OPT_GRAPH, 1)
    return state


def run(state):
    ctx = state["ctx"]
    if state["kind"] == "3d":
        return dict(zip(("phi", "ex", "ey", "ez"), ctx.evaluate(*state["args"])))
    if state["kind"] == "batch":
        ctx.evaluate_batch(state["items"])
        return state["out"]
    if state["kind"] == "host":
        out = state["out"]
        ctx.evaluate_host_ptrs(out["u"].numel(), *(t.data_ptr() for t in state["args"]),
                               out["u"].data_ptr(), out["v"].data_ptr())
        return out
    u, v = ctx.evaluate(*state["args"])
    return {"u": u, "v": v}


# --------------------------------------------------------------------------- what a pass needs

def work(case):
    """Inputs read once and outputs written once; the flops of the expansions (8 p per blob in
    and out, 8 p^2 per translation, 27 or 189 a box) and of the near field, each unordered pair
    once.  A blob core wider than a leaf makes the near kernel smooth, so there a blob needs no
    more than one more expansion in and out."""
    c = case
    size = 4 if c["dtype"] == "f32" else 8
    if c["kind"] == "batch":
        flops = 0.0
        for n, p in zip(*(v.tolist() for v in _batch_sizes(c))):
            flops += _flops2(n, p, 9.0 * 16, n / 16, False)
        return {"bytes": 5.0 * size * _count(c), "flops": flops}
    n, p, boxes = _count(c), c["p"], float((8 if c["kind"].endswith("3d") else 4) ** c["L"])
    near = n / boxes  # blobs per leaf as a blob meets them
    if c["kind"] == "clustered":
        near *= 1.0 / (8 * 4 * math.pi * 0.02 ** 2)
    elif c["kind"] == "clustered3d":
        near *= 1.0 / (8 * (4 * math.pi * 0.04 ** 2) ** 1.5)
    boxes = min(boxes, float(n), n / near)
    if c["kind"].endswith("3d"):
        pairs = 0.5 * 27 * near * n
        return {"bytes": 8.0 * size * n,
                "flops": 26 * pairs + 4.0 * p * p * n + 189 * 8 / 7 * boxes * 2 * p ** 4}
    width = 2 * (c["half_width"] + 0.8 * c["sigma"]) if c["kind"] == "lamb_oseen" else 1.0
    smooth = "sigma" in c and c["sigma"] >= width / 2 ** c["L"]
    return {"bytes": 5.0 * size * n, "flops": _flops2(n, p, 9 * near, boxes, smooth)}


def _flops2(n, p, neighbours, boxes, smooth):
    pair = 0.5 * 14 * neighbours
    if smooth:
        pair = min(pair, 16.0 * p)
    return n * (16.0 * p + pair) + 27 * 4 / 3 * boxes * 8 * p * p


def exact(case, seed):
    """The sums the evaluation approximates, in FP64: near pairs (leaves that touch) with the
    blob kernel and the others with the singular kernel, as the method defines its result."""
    c = case
    if c["kind"] == "batch":
        return None  # hours of pairs
    n = _count(c)
    if n > (1 << 18 if c["kind"].endswith("3d") else 1 << 17):
        return None
    xs, q, sigma, domain = _inputs(c, seed)
    xs, q = [v.double() for v in xs], q.double()
    step = max(1, (1 << 27) // n)
    out = []
    for i in range(0, n, step):
        d = [v[i:i + step, None] - v[None, :] for v in xs]
        r2 = sum(v * v for v in d)
        same = r2 == 0
        r2[same] = 1.0
        if c["kind"].endswith("3d"):
            w = q / r2.sqrt()
            w[same] = 0.0
            f = w / r2
            out.append([w.sum(1)] + [(f * v).sum(1) for v in d])
        elif c["kind"] == "laplace":
            out.append([0.5 * (r2.log() @ q)])
        else:
            cell = [((v - o) * (2 ** c["L"] / domain[-1])).floor().clamp(0, 2 ** c["L"] - 1)
                    for v, o in zip(xs, domain)]
            far = torch.zeros_like(same)
            for v in cell:
                far |= (v[i:i + step, None] - v[None, :]).abs() > 1
            k = torch.where(far, 1.0, -torch.expm1(r2 * (-0.5 / sigma ** 2)))
            k = k * (q / (2 * math.pi)) / r2
            k[same] = 0.0
            out.append([-(k * d[1]).sum(1), (k * d[0]).sum(1)])
    out = [torch.cat(v) for v in zip(*out)]
    if c["kind"] == "laplace":
        return {"u": out[0], "v": torch.zeros_like(out[0])}
    names = ("phi", "ex", "ey", "ez") if c["kind"].endswith("3d") else ("u", "v")
    if c.get("host"):
        out = [v.cpu() for v in out]
    return dict(zip(names, out))
