"""The work that users of this max-flow solver have it do, as cases to be timed: single graphs that stay on the GPU and are solved
through ``mf.Graph``, batches (``mf.Batch``) and bursts of requests to a running service (``mf.Service``).

The families are those of ``paper_1507_01926_gb300/inputs`` (2D image grids, multi-frame video grids, 3D volume grids, R-MAT power-law
graphs, layered random graphs) with the same structure and capacity ranges, drawn here on the GPU so that inputs are made quickly.

Every solve writes the flow value, the per-slot flow (unless the case asks for the cut only) and the minimal source-side cut. A maximum
flow is not unique, and the default rounds give another one on every solve, so ``run`` returns the value and the cut, which are unique;
with ``simple_rounds`` the flow is the same on every solve and is returned as well. All outputs are whole numbers: there is nothing for
``exact`` to say about rounding.
"""
import math
import random

import numpy as np
import torch

from paper_1507_01926_gb300 import mf

VOLUME = (256, 256, 128)

# The packaged autotuner choices for the three tuned workloads of the benchmark, as a user applies them.
TUNED = {
    "grid3d": {"gr_time_ratio": 4.0, "bfs_hops": 4},
    "rmat": {"gr_time_ratio": 4.0, "gr_freq": 1.0, "bin_warp": 128, "blocks_per_sm": 2, "kernel_variant": 1, "bfs_pull": 50},
    "layered": {"gr_time_ratio": 4.0, "bin_thread": 16, "block_threads": 64, "blocks_per_sm": 4, "kernel_variant": 4, "bfs_pull": 20},
}


def listed():
    return [
        # a thumbnail or one region of an image: the smallest call, where launch and barrier latency counts
        {"name": "image-64", "kind": "grid2d", "h": 64, "w": 64},
        # foreground / background segmentation of a photograph: only the cut is wanted, handed to the host
        {"name": "segment-321x481", "kind": "grid2d", "h": 321, "w": 481, "cut_only": True},
        # the largest image of the serving workload, with its flow
        {"name": "image-1024", "kind": "grid2d", "h": 1024, "w": 1024},
        # reproducible per-arc flow on an image
        {"name": "image-det-150x211", "kind": "grid2d", "h": 150, "w": 211, "simple": True},
        # segmentation through a short video: frames coupled by motion arcs
        {"name": "video-24", "kind": "frames", "f": 24, "side": 128},
        # a small volume of odd sides with default options
        {"name": "volume-97x80x61", "kind": "grid3d", "x": 97, "y": 80, "z": 61},
        # the benchmark's volume with the packaged tuned options
        {"name": "volume-256x256x128", "kind": "grid3d", "x": VOLUME[0], "y": VOLUME[1], "z": VOLUME[2], "tuned": True},
        # a web-like power-law graph with the packaged tuned options
        {"name": "web-s22", "kind": "rmat", "scale": 22, "ef": 16, "tuned": True},
        # one layered random graph (average degree 10) with default options
        {"name": "layers-96x700", "kind": "layered", "layers": 96, "width": 700},
        # many uneven layered graphs solved by one launch with the packaged tuned options
        {"name": "batch-40", "kind": "batch", "count": 40, "sizes": 3, "tuned": True},
        # a burst of image and video requests to a running service
        {"name": "service-24", "kind": "service", "count": 24, "sizes": 1},
    ]


def _log_uniform(rng, a, b):
    return min(b, max(a, int(math.exp(rng.uniform(math.log(a), math.log(b + 1))))))


def draw(rng):
    kind = rng.choice(["grid2d", "grid2d", "cut", "det", "frames", "grid3d", "grid3d", "rmat", "layered", "batch", "service"])
    if kind in ("grid2d", "cut", "det"):
        top = 1024 if kind != "det" else 256
        case = {"kind": "grid2d", "h": _log_uniform(rng, 32, top), "w": _log_uniform(rng, 32, top)}
        if kind == "cut":
            case["cut_only"] = True
        if kind == "det":
            case["simple"] = True
        return case
    if kind == "frames":
        return {"kind": "frames", "f": rng.randint(4, 64), "side": rng.choice([64, 96, 128, 131])}
    if kind == "grid3d":
        return {"kind": "grid3d", "x": _log_uniform(rng, 16, 256), "y": _log_uniform(rng, 16, 256), "z": _log_uniform(rng, 16, 128),
                "tuned": rng.random() < 0.5}
    if kind == "rmat":
        return {"kind": "rmat", "scale": rng.randint(12, 22), "ef": rng.choice([8, 11, 16]), "tuned": rng.random() < 0.5}
    if kind == "layered":
        return {"kind": "layered", "layers": _log_uniform(rng, 16, 256), "width": _log_uniform(rng, 64, 2048)}
    return {"kind": kind, "count": rng.randint(8, 40 if kind == "batch" else 24), "sizes": rng.randint(0, 1 << 20),
            **({"tuned": rng.random() < 0.5} if kind == "batch" else {})}


# ---------------------------------------------------------------- instances, made on the GPU

def _caps(gen, n, lo, hi):
    return torch.randint(lo, hi + 1, (n,), generator=gen, device="cuda", dtype=torch.int32)


def _csr(n, u, v, cuv, cvu):
    """Paired-slot CSR of the vertex pairs (u, v) with capacities u->v and v->u: int64 row offsets, int32 head and cap, int64 rev, the
    rows sorted by head."""
    p = u.numel()
    tail, head, cap = torch.cat([u, v]), torch.cat([v, u]), torch.cat([cuv, cvu])
    _, order = torch.sort(tail * n + head, stable=True)
    place = torch.empty_like(order)
    place[order] = torch.arange(2 * p, device="cuda")
    rev = place[torch.where(order < p, order + p, order - p)]
    row = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    row[1:] = torch.cumsum(torch.bincount(tail, minlength=n), 0)
    return row, head[order].to(torch.int32), cap[order].contiguous(), rev


def _lattice(dims):
    """Neighbour pairs of a lattice, dims from the slowest to the fastest axis, numbered in row-major order."""
    idx = torch.arange(math.prod(dims), device="cuda").view(dims)
    us, vs = [], []
    for d in range(len(dims)):
        us.append(idx.narrow(d, 0, dims[d] - 1).reshape(-1))
        vs.append(idx.narrow(d, 1, dims[d] - 1).reshape(-1))
    return torch.cat(us), torch.cat(vs)


def _pixel_terminals(gen, np_, s, t):
    """Every pixel gets s->p with probability 1/2, else p->t, capacity U[1,1000]."""
    p = torch.arange(np_, device="cuda")
    c = _caps(gen, np_, 1, 1000)
    src = torch.rand(np_, generator=gen, device="cuda") < 0.5
    z = torch.zeros_like(c)
    return torch.where(src, s, p), torch.where(src, p, t), c, z


def _grid2d(gen, h, w):
    u, v = _lattice((h, w))
    n = h * w
    a, b, c, z = _pixel_terminals(gen, n, n, n + 1)
    k = u.numel()
    return n + 2, n, n + 1, _csr(n + 2, torch.cat([u, a]), torch.cat([v, b]), torch.cat([_caps(gen, k, 1, 100), c]),
                                torch.cat([_caps(gen, k, 1, 100), z]))


def _frames(gen, f, side):
    fp = side * side
    u0, v0 = _lattice((side, side))
    at = (torch.arange(f, device="cuda") * fp).view(f, 1)
    u, v = (u0 + at).reshape(-1), (v0 + at).reshape(-1)
    k, n = u.numel(), f * fp
    perm = torch.argsort(torch.rand((f - 1, fp), generator=gen, device="cuda"), dim=1)
    mu = torch.arange(n - fp, device="cuda")
    mv = (perm + at[1:]).reshape(-1)
    a, b, c, z = _pixel_terminals(gen, n, n, n + 1)
    return n + 2, n, n + 1, _csr(n + 2, torch.cat([u, mu, a]), torch.cat([v, mv, b]),
                                torch.cat([_caps(gen, k, 1, 1000), _caps(gen, n - fp, 1, 100), c]),
                                torch.cat([_caps(gen, k, 1, 1000), torch.zeros(n - fp, dtype=torch.int32, device="cuda"), z]))


def _grid3d(gen, x, y, z):
    u, v = _lattice((z, y, x))
    n, face, k = x * y * z, x * y, u.numel()
    p = torch.arange(face, device="cuda")
    big = torch.full((2 * face,), 1_000_000, dtype=torch.int32, device="cuda")
    a = torch.cat([torch.full_like(p, n), p + (n - face)])
    b = torch.cat([p, torch.full_like(p, n + 1)])
    return n + 2, n, n + 1, _csr(n + 2, torch.cat([u, a]), torch.cat([v, b]), torch.cat([_caps(gen, k, 1, 1000), big]),
                                torch.cat([_caps(gen, k, 1, 1000), torch.zeros_like(big)]))


def _rmat(gen, scale, ef):
    """R-MAT (0.57, 0.19, 0.19, 0.05), self-loops and repeats dropped, an arc and its opposite in one pair; s is the vertex of largest
    out-degree, t that of largest in-degree among the rest."""
    n, d = 1 << scale, ef << scale
    u = torch.zeros(d, dtype=torch.int64, device="cuda")
    v = torch.zeros(d, dtype=torch.int64, device="cuda")
    for _ in range(scale):
        q = torch.rand(d, generator=gen, device="cuda")
        u = u * 2 + (q >= 0.76)
        v = v * 2 + (((q >= 0.57) & (q < 0.76)) | (q >= 0.95))
    key = torch.unique((u * n + v)[u != v])
    u, v = key // n, key % n
    cap = _caps(gen, u.numel(), 1, 1000)
    low = torch.arange(n - 1, -1, -1, device="cuda")
    s = int(n - 1 - (torch.bincount(u, minlength=n) * n + low).max() % n)
    ind = torch.bincount(v, minlength=n)
    ind[s] = -1
    t = int(n - 1 - (ind * n + low).max() % n)
    pair, at = torch.unique(torch.minimum(u, v) * n + torch.maximum(u, v), return_inverse=True)
    cuv = torch.zeros(pair.numel(), dtype=torch.int32, device="cuda")
    cvu = torch.zeros_like(cuv)
    up = u < v
    cuv[at[up]] = cap[up]
    cvu[at[~up]] = cap[~up]
    return n, s, t, _csr(n, pair // n, pair % n, cuv, cvu)


def _layered(gen, layers, width):
    """4 arcs from every vertex to uniform vertices of the next layer, 1 to another vertex of its layer, capacity U[1,10000]."""
    n = layers * width
    p = torch.arange(n - width, device="cuda")
    u = p.repeat_interleave(4)
    v = (u // width + 1) * width + torch.randint(0, width, (u.numel(),), generator=gen, device="cuda")
    q = torch.arange(n, device="cuda")
    r = torch.randint(1, width, (n,), generator=gen, device="cuda")
    w = q // width * width + (q % width + r) % width
    j = torch.arange(width, device="cuda")
    k = u.numel() + n
    a = torch.cat([torch.full_like(j, n), j + (n - width)])
    b = torch.cat([j, torch.full_like(j, n + 1)])
    cap = torch.cat([_caps(gen, k, 1, 10000), torch.full((2 * width,), 1_000_000, dtype=torch.int32, device="cuda")])
    return n + 2, n, n + 1, _csr(n + 2, torch.cat([u, q, a]), torch.cat([v, w, b]), cap, torch.zeros_like(cap))


def _members(case):
    """Sizes of the instances of a batch or a burst: layered graphs as (layers, width), requests as ("grid", side) or ("frames", f)."""
    rng = random.Random(case["sizes"])
    if case["kind"] == "batch":
        return [(_log_uniform(rng, 16, 256), _log_uniform(rng, 64, 1024)) for _ in range(case["count"])]
    return [("grid", _log_uniform(rng, 32, 512)) if rng.random() < 0.5 else ("frames", rng.randint(4, 16)) for _ in range(case["count"])]


def _options(case, default):
    o = default()
    if case.get("tuned"):
        for k, v in TUNED["layered" if case["kind"] == "batch" else case["kind"]].items():
            setattr(o, k, v)
    o.cut_only = 1 if case.get("cut_only") else 0
    o.simple_rounds = 1 if case.get("simple") else 0
    return o


def _host(inst):
    n, s, t, (row, head, cap, rev) = inst
    return mf.CSR(n, row.cpu().numpy(), head.cpu().numpy(), cap.cpu().numpy(), rev.cpu().numpy(), np.zeros(0, np.int64), 0), (s, t)


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    kind = case["kind"]
    if kind in ("batch", "service"):
        made = []
        for a, b in _members(case):
            made.append(_host(_layered(gen, a, b) if kind == "batch" else _grid2d(gen, b, b) if a == "grid" else _frames(gen, b, 128)))
        csrs, ends = [m[0] for m in made], [m[1] for m in made]
        if kind == "batch":
            return {"kind": kind, "batch": mf.Batch(csrs, ends, _options(case, mf.default_options))}
        return {"kind": kind, "service": mf.Service(8 << 30), "requests": list(zip(csrs, ends))}
    if kind == "grid2d":
        n, s, t, csr = _grid2d(gen, case["h"], case["w"])
    elif kind == "frames":
        n, s, t, csr = _frames(gen, case["f"], case["side"])
    elif kind == "grid3d":
        n, s, t, csr = _grid3d(gen, case["x"], case["y"], case["z"])
    elif kind == "rmat":
        n, s, t, csr = _rmat(gen, case["scale"], case["ef"])
    else:
        n, s, t, csr = _layered(gen, case["layers"], case["width"])
    graph = mf.Graph.from_device(n, *csr, s, t, _options(case, mf.default_options))
    if case.get("cut_only"):
        return {"kind": "cut", "graph": graph}
    return {"kind": "det" if case.get("simple") else "graph", "graph": graph,
            "value": torch.zeros(1, dtype=torch.int64, device="cuda"),
            "flow": torch.zeros(graph.m, dtype=torch.int32, device="cuda"),
            "cut": torch.zeros((n + 31) // 32, dtype=torch.int32, device="cuda")}


def run(state):
    kind = state["kind"]
    if kind == "batch":
        got = state["batch"].solve(flow=False, cut=True)
        return {"values": np.array([r.value for r in got], np.int64), "cuts": np.concatenate([r.cut_bits for r in got]).view(np.int32)}
    if kind == "service":
        service = state["service"]
        tickets = [service.submit(csr, s, t) for csr, (s, t) in state["requests"]]
        got = []
        for k in tickets:
            service.wait(k)
            got.append(service.poll(k))
        return {"values": np.array([r.value for r in got], np.int64), "cuts": np.concatenate([r.cut_bits for r in got]).view(np.int32)}
    if kind == "cut":
        got = state["graph"].solve(flow=False, cut=True)
        return {"value": got.value, "cut": got.cut_bits.view(np.int32)}
    state["graph"].solve_device(state["value"], state["flow"], state["cut"])
    out = {"value": state["value"], "cut": state["cut"]}
    if kind == "det":
        out["flow"] = state["flow"]
    return out


def _size(kind, case):
    """Vertices and slots (two for each vertex pair with an arc)."""
    if kind == "grid2d":
        h, w = case
        return h * w + 2, 2 * (h * (w - 1) + w * (h - 1) + h * w)
    if kind == "frames":
        f, side = case
        fp = side * side
        return f * fp + 2, 2 * (2 * f * side * (side - 1) + (f - 1) * fp + f * fp)
    if kind == "grid3d":
        x, y, z = case
        return x * y * z + 2, 2 * ((x - 1) * y * z + x * (y - 1) * z + x * y * (z - 1) + 2 * x * y)
    if kind == "rmat":
        scale, ef = case
        return 1 << scale, 2 * (ef << scale)
    layers, width = case
    return layers * width + 2, 2 * (4 * (layers - 1) * width + layers * width + 2 * width)


def work(case):
    """One pass reads the graph once (4 bytes for each row offset and 12 for each slot's head, reverse slot and capacity) and writes
    the cut's bits, the value and, where it is asked for, 4 bytes of flow for each slot. How often push-relabel has to visit a vertex
    is not known in advance, so this is the least, not what any known algorithm reaches."""
    kind = case["kind"]
    flow = not case.get("cut_only") and kind != "batch"
    if kind == "batch":
        sizes = [_size("layered", m) for m in _members(case)]
    elif kind == "service":
        sizes = [_size("grid2d", (m[1], m[1])) if m[0] == "grid" else _size("frames", (m[1], 128)) for m in _members(case)]
    else:
        keys = {"grid2d": ("h", "w"), "frames": ("f", "side"), "grid3d": ("x", "y", "z"), "rmat": ("scale", "ef"), "layered": ("layers", "width")}
        sizes = [_size(kind, tuple(case[k] for k in keys[kind]))]
    return {"bytes": sum(4 * (n + 1) + 12 * m + n // 8 + 8 + (4 * m if flow else 0) for n, m in sizes), "flops": 0}


def exact(case, seed):
    """Values, cuts and flows are whole numbers, equal for every correct solve: there is no rounding to compare."""
    return None
