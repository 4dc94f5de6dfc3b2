"""Which solver a call runs and what it leaves behind, for single 2D and 3D grids (the lattice solvers) and graphs
that are nearly such grids (the list solver). A lattice solve counts no rounds by size, a list solve does."""
import numpy as np
import pytest

import oracle
from paper_1507_01926_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def grid(dims, seed):
    """A lattice whose cells all have an arc from s or to t (side lengths from the slowest axis to the fastest)."""
    rng = np.random.default_rng(seed)
    idx = np.arange(int(np.prod(dims))).reshape(dims)
    u = np.concatenate([np.take(idx, np.arange(d - 1), axis=k).ravel() for k, d in enumerate(dims)])
    v = np.concatenate([np.take(idx, np.arange(1, d), axis=k).ravel() for k, d in enumerate(dims)])
    n = idx.size
    src = rng.random(n) < 0.5
    cells = np.arange(n)
    tail = np.concatenate([u, v, np.where(src, n, cells)])
    head = np.concatenate([v, u, np.where(src, cells, n + 1)])
    cap = np.concatenate([rng.integers(1, 101, 2 * u.size), rng.integers(1, 201, n)])
    return I.Instance(n + 2, n, n + 1, tail.astype(np.int32), head.astype(np.int32), cap.astype(np.int32), f"grid_{dims}")


def on_lattice(stats):
    return stats["rounds"] > 0 and not any(stats["rounds_by_size"])


def on_lists(stats):
    return any(stats["rounds_by_size"])


def add_self_loop(csr, v):
    """The CSR with one more slot pair v -> v at the end of v's row."""
    at = int(csr.row_offsets[v + 1])
    row = csr.row_offsets.copy()
    row[v + 1:] += 2
    rev = csr.rev + 2 * (csr.rev >= at)
    return (row, np.insert(csr.head, at, [v, v]).astype(np.int32), np.insert(csr.cap, at, [3, 4]).astype(np.int32),
            np.insert(rev, at, [at + 1, at]).astype(np.int64), at)


DIMS = [(20, 33), (9, 10, 11)]


@pytest.mark.parametrize("dims", DIMS)
@pytest.mark.parametrize("where", ["s", "t", "cell"])
def test_self_loops_have_their_flow_written(gpu, dims, where):
    """A raw CSR may hold slot pairs from a vertex to itself (mf_build_csr drops them): the graph is no lattice, and
    every slot of the flow output is written."""
    import torch

    g = grid(dims, 1)
    csr = gpu.build_csr(g.n, g.tail, g.head, g.cap)
    row, head, cap, rev, at = add_self_loop(csr, {"s": g.s, "t": g.t, "cell": 7}[where])
    dev = torch.device("cuda", 0)
    st = torch.cuda.Stream()
    arrays = [torch.from_numpy(a).to(dev) for a in (row, head, cap, rev)]
    val = torch.zeros(1, dtype=torch.int64, device=dev)
    flow = torch.full((head.size,), -7, dtype=torch.int32, device=dev)
    cut = torch.zeros((g.n + 31) // 32, dtype=torch.int32, device=dev)
    torch.cuda.synchronize()
    G = gpu.Graph.from_device(g.n, *arrays, g.s, g.t, stream=st)
    try:
        G.solve_device(val, flow, cut, stream=st)
        stats = G.stats()
    finally:
        G.close()
    ref = oracle.maxflow(g.n, g.s, g.t, g.tail, g.head, g.cap, want_flow=False)
    f = flow.cpu().numpy()
    assert int(val.item()) == ref["value"]
    assert np.array_equal(gpu.cut_bits_to_bool(cut.cpu().numpy().view(np.uint32), g.n), ref["cut"])
    assert f[at] == 0 and f[at + 1] == 0 and f.min() >= 0
    assert on_lists(stats)


def test_capture_follows_the_launch_shape(gpu):
    """A replayed solve takes a new blocks_per_sm, as a direct launch does."""
    g = grid((700, 512), 2)  # 704 tiles
    csr = gpu.build_csr(g.n, g.tail, g.head, g.cap)

    def shapes(use_graph):
        got = []
        with gpu.Graph.from_csr(csr, g.s, g.t) as G:
            for bps in (4, 3, 2, 4):
                G.set_options(gpu.default_options(use_graph=use_graph, blocks_per_sm=bps))
                value = G.solve(flow=False).value
                assert on_lattice(G.stats())
                got.append((value, G.stats()["grid_blocks"]))
        return got

    assert shapes(1) == shapes(0)


def test_unions_of_one_are_not_prepared_as_lattices(gpu):
    """Batches and services run the list solver: a one-member union of a thin grid (whose padded tiles are several
    times its cells) allocates no tiles."""
    import torch

    g = grid((60000, 5), 3)
    csr = gpu.build_csr(g.n, g.tail, g.head, g.cap)
    other = gpu.build_csr(g.n, np.append(g.tail, g.s), np.append(g.head, g.t), np.append(g.cap, 5).astype(np.int32))
    used = []
    with gpu.Batch([other], [(g.s, g.t)]):  # the library's code is on the device before memory is looked at
        pass
    for c in (csr, other):  # the second is no lattice
        torch.cuda.synchronize()
        before = torch.cuda.mem_get_info()[0]
        with gpu.Batch([c], [(g.s, g.t)]):
            used.append(before - torch.cuda.mem_get_info()[0])
    assert abs(used[0] - used[1]) <= 8 << 20, used


def test_autotune_of_a_lattice_moves_only_what_it_reads(gpu):
    """Options that a lattice solve does not read are not tuned by the noise between identical solves."""
    g = grid((300, 260), 4)
    csr = gpu.build_csr(g.n, g.tail, g.head, g.cap)
    start = gpu.default_options()
    with gpu.Graph.from_csr(csr, g.s, g.t, start) as G:
        value = G.solve(flow=False).value
        best, ms = G.autotune(reps=1, sweeps=2)
        assert G.solve(flow=False).value == value and on_lattice(G.stats())
    d, s = gpu.options_to_dict(best), gpu.options_to_dict(start)
    assert {k for k in d if d[k] != s[k]} <= {"gr_time_ratio", "blocks_per_sm"}


@pytest.mark.parametrize("dims,lattice", [((2, 60000), True), ((2, 140000), False), ((40005, 8), True), ((40000, 7), False),
                                          ((4, 5, 20000), True), ((3, 4, 40000), False), ((200, 3), True)])
def test_thin_boxes_take_the_faster_solver(gpu, dims, lattice):
    """More than 2,048 tiles that are mostly padding are left to the list solver."""
    g = grid(dims, 5)
    csr = gpu.build_csr(g.n, g.tail, g.head, g.cap)
    ref = oracle.maxflow(g.n, g.s, g.t, g.tail, g.head, g.cap, want_flow=False)
    with gpu.Graph.from_csr(csr, g.s, g.t) as G:
        r = G.solve()
        assert on_lattice(G.stats()) == lattice
    cut = gpu.cut_bits_to_bool(r.cut_bits, g.n)
    assert r.value == ref["value"] and np.array_equal(cut, ref["cut"])
    f = np.where(csr.arc_slot >= 0, r.flow[np.maximum(csr.arc_slot, 0)], 0).astype(np.int64)
    assert not oracle.check_flow(g.n, g.s, g.t, g.tail, g.head, g.cap, f, r.value, cut)


def test_tiles_take_memory_only_while_options_use_them(gpu):
    """A thin grid's tiles are in a buffer of their own (here some 50 MB); a graph whose options keep it on the
    list solver has none, and where the device has no room for an output they give way to it."""
    import torch

    g = grid((40000, 8), 6)
    csr = gpu.build_csr(g.n, g.tail, g.head, g.cap)
    lists = dict(max_rounds=2_000_000)  # the default limit, named: a list solve
    small = grid((40, 30), 7)
    warm = gpu.build_csr(small.n, small.tail, small.head, small.cap)
    for o in ({}, lists):  # both solvers' code is on the device before memory is looked at
        with gpu.Graph.from_csr(warm, small.s, small.t, gpu.default_options(**o)) as G:
            G.solve()
    torch.cuda.synchronize()

    def free():
        return torch.cuda.mem_get_info()[0]

    before = free()
    with gpu.Graph.from_csr(csr, g.s, g.t, gpu.default_options(**lists)) as G:
        plain = before - free()
        value = G.solve(flow=False, cut=False).value
        assert on_lists(G.stats())
        G.set_options(gpu.default_options())
        tiled = before - free()
        assert G.solve(flow=False, cut=False).value == value and on_lattice(G.stats())
        assert tiled - plain >= 32 << 20
        G.set_options(gpu.default_options(**lists))
        assert before - free() <= plain + (4 << 20)
        G.set_options(gpu.default_options())
        torch.cuda.empty_cache()
        rest = torch.empty(free() - (4 << 20), dtype=torch.uint8, device="cuda")  # leaves less than the flow needs
        assert free() < 4 * G.m
        try:
            r = G.solve()
        finally:
            del rest
            torch.cuda.empty_cache()
        assert r.value == value and on_lists(G.stats())
    f = np.where(csr.arc_slot >= 0, r.flow[np.maximum(csr.arc_slot, 0)], 0).astype(np.int64)
    cut = gpu.cut_bits_to_bool(r.cut_bits, g.n)
    assert not oracle.check_flow(g.n, g.s, g.t, g.tail, g.head, g.cap, f, r.value, cut)


@pytest.mark.parametrize("opts", [{}, dict(cut_only=1), dict(use_graph=1)])
@pytest.mark.parametrize("dims", [(150, 130), (20, 30, 25)])
def test_solves_that_are_given_up_end_on_the_list_solver(gpu, dims, opts):
    """With the lattice kernels built to give up after a few sweeps or visits, every solve still has its result."""
    from paper_1507_01926_gb300 import build as mfbuild

    g = grid(dims, 8)
    csr = gpu.build_csr(g.n, g.tail, g.head, g.cap)
    ref = oracle.maxflow(g.n, g.s, g.t, g.tail, g.head, g.cap, want_flow=False)
    before = gpu.use_library(mfbuild.build_limit())
    try:
        with gpu.Graph.from_csr(csr, g.s, g.t, gpu.default_options(**opts)) as G:
            for _ in range(2):
                r = G.solve(flow=not opts.get("cut_only"))
                assert on_lists(G.stats())
                cut = gpu.cut_bits_to_bool(r.cut_bits, g.n)
                assert r.value == ref["value"] and np.array_equal(cut, ref["cut"])
                if r.flow is not None:
                    f = np.where(csr.arc_slot >= 0, r.flow[np.maximum(csr.arc_slot, 0)], 0).astype(np.int64)
                    assert not oracle.check_flow(g.n, g.s, g.t, g.tail, g.head, g.cap, f, r.value, cut)
    finally:
        gpu.use_library(before)


@pytest.mark.parametrize("cut_only", [0, 1])
def test_volume_scans_count_slots_that_exist(gpu, cut_only):
    """Arcs along the slowest axis only (and one along each other, which make the box known): a cell has at most two
    slots to neighbours and one to a terminal; four cells have one more."""
    dims = (20, 24, 22)
    g = grid(dims, 9)
    cell = (g.tail < g.s) & (g.head < g.s)
    step = np.where(cell, np.abs(g.tail - g.head), 0)
    keep = ~cell | (step == 24 * 22)
    for k in (1, 22):
        keep[np.flatnonzero(step == k)[0]] = True
    csr = gpu.build_csr(g.n, g.tail[keep], g.head[keep], g.cap[keep])
    with gpu.Graph.from_csr(csr, g.s, g.t, gpu.default_options(cut_only=cut_only)) as G:
        G.solve(flow=False)
        st = G.stats()
    assert on_lattice(st) and st["visits_discharge"] > 0 and st["visits_bfs"] > 0
    assert st["scans_discharge"] <= 3 * st["visits_discharge"] + 4 * 16 * st["rounds"]  # 16 rounds a visit at most
    assert 0 < st["scans_discharge_residual"] <= st["scans_discharge"]
    assert st["scans_bfs"] <= 2.1 * st["visits_bfs"]


@pytest.mark.parametrize("opts", [{}, dict(cut_only=1), dict(gr_time_ratio=1e-6)])
@pytest.mark.parametrize("dims", [(40, 37), (17, 33), (400, 3), (20, 18, 12), (9, 17, 7), (3, 4, 60)])
def test_checked_build_runs_the_lattice_kernels(gpu, dims, opts):
    """The build with checked gathers solves lattices by the lattice kernels, and finds no index out of bounds."""
    from paper_1507_01926_gb300 import build as mfbuild

    g = grid(dims, 10)
    csr = gpu.build_csr(g.n, g.tail, g.head, g.cap)
    ref = oracle.maxflow(g.n, g.s, g.t, g.tail, g.head, g.cap, want_flow=False)
    before = gpu.use_library(mfbuild.build(check=True))
    try:
        with gpu.Graph.from_csr(csr, g.s, g.t, gpu.default_options(**opts)) as G:
            r = G.solve(flow=not opts.get("cut_only"))
            assert on_lattice(G.stats())
    finally:
        gpu.use_library(before)
    cut = gpu.cut_bits_to_bool(r.cut_bits, g.n)
    assert r.value == ref["value"] and np.array_equal(cut, ref["cut"])
    if r.flow is not None:
        f = np.where(csr.arc_slot >= 0, r.flow[np.maximum(csr.arc_slot, 0)], 0).astype(np.int64)
        assert not oracle.check_flow(g.n, g.s, g.t, g.tail, g.head, g.cap, f, r.value, cut)
