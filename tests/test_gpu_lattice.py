"""The lattice solvers (single graphs whose vertices are the cells of a 2D or 3D box): tiles of 32 x 16 and
8 x 8 x 8 cells. Sizes at the edges of tiles, boxes with a cut-short last row or plane, terminals anywhere in the
numbering, capacities up to the int32 limit and empty or full ones; and graphs that are almost lattices, which the
list solver takes. Value and S_min are unique and must equal the oracle's; the flow must satisfy its definitions."""
import numpy as np
import pytest

import oracle
from paper_1507_01926_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def box(dims, seed, cap=(1, 100), term=(0, 200), keep=1.0, cells=None, s_at=None, t_at=None, tweak=None):
    """A lattice with the given side lengths (slowest axis first), of which the first `cells` cells exist; every
    cell gets an arc from s or to t; s and t are inserted at positions s_at and t_at of the numbering."""
    rng = np.random.default_rng(seed)
    n = int(np.prod(dims)) if cells is None else cells
    idx = np.arange(int(np.prod(dims))).reshape(dims)
    us, vs = [], []
    for d in range(len(dims)):
        u = np.take(idx, np.arange(dims[d] - 1), axis=d).ravel()
        v = np.take(idx, np.arange(1, dims[d]), axis=d).ravel()
        us.append(u)
        vs.append(v)
    u, v = np.concatenate(us), np.concatenate(vs)
    k = (u < n) & (v < n) & (rng.random(u.size) < keep)
    u, v = u[k], v[k]
    lo, hi = sorted((n if s_at is None else s_at, n + 1 if t_at is None else t_at))
    vert = np.arange(n)
    vert = vert + (vert >= lo)
    vert = vert + (vert >= hi)
    s, t = (n if s_at is None else s_at), (n + 1 if t_at is None else t_at)
    src = rng.random(n) < 0.5
    tail = np.concatenate([vert[u], vert[v], np.where(src, s, vert)])
    head = np.concatenate([vert[v], vert[u], np.where(src, vert, t)])
    c = np.concatenate([rng.integers(cap[0], cap[1] + 1, 2 * u.size), rng.integers(term[0], term[1] + 1, n)])
    if tweak:
        tail, head, c = tweak(tail, head, c, vert, s, t)
    return I.Instance(n + 2, int(s), int(t), tail.astype(np.int32), head.astype(np.int32), c.astype(np.int32),
                      f"box_{dims}_{seed}")


def check(gpu, g, **opts):
    csr = gpu.build_csr(g.n, g.tail, g.head, g.cap)
    ref = oracle.maxflow(g.n, g.s, g.t, g.tail, g.head, g.cap, want_flow=False)
    with gpu.Graph.from_csr(csr, g.s, g.t, gpu.default_options(**opts)) as G:
        for _ in range(2):  # a solve starts from the capacities, whatever the last one left
            r = G.solve(flow=not opts.get("cut_only"))
            cut = gpu.cut_bits_to_bool(r.cut_bits, g.n)
            assert r.value == ref["value"], g.name
            assert np.array_equal(cut, ref["cut"]), g.name
            if not opts.get("cut_only"):
                f = np.where(csr.arc_slot >= 0, r.flow[np.maximum(csr.arc_slot, 0)], 0).astype(np.int64)
                assert not oracle.check_flow(g.n, g.s, g.t, g.tail, g.head, g.cap, f, r.value, cut), g.name


@pytest.mark.parametrize("dims", [(2, 2), (15, 31), (16, 32), (17, 33), (3, 64), (50, 5), (33, 97), (130, 70),
                                  (2, 2, 2), (7, 8, 9), (8, 8, 8), (9, 17, 7), (16, 16, 16), (3, 40, 5), (25, 31, 18)])
@pytest.mark.parametrize("cut_only", [0, 1])
def test_tile_edges(gpu, dims, cut_only):
    check(gpu, box(dims, sum(dims)), cut_only=cut_only)


@pytest.mark.parametrize("dims,cells", [((20, 33), 20 * 33 - 20), ((9, 10, 11), 9 * 110 - 57), ((6, 9, 8), 6 * 72 - 8)])
def test_cut_short_boxes_and_terminals_inside(gpu, dims, cells):
    check(gpu, box(dims, 5, cells=cells))
    check(gpu, box(dims, 6, cells=cells, s_at=0, t_at=cells // 2))
    check(gpu, box(dims, 7, cells=cells, s_at=cells // 3, t_at=1, keep=0.7))


@pytest.mark.parametrize("dims", [(40, 40), (12, 13, 14)])
def test_capacities(gpu, dims):
    big = 2 ** 30 - 1  # a pair's capacities sum to INT32_MAX - 1
    check(gpu, box(dims, 11, cap=(big - 9, big), term=(2 ** 31 - 99, 2 ** 31 - 1)))  # excess beyond int32
    check(gpu, box(dims, 12, cap=(0, 2), term=(0, 2 ** 31 - 1)))
    check(gpu, box(dims, 13, cap=(0, 0)))
    check(gpu, box(dims, 14, term=(0, 0)))
    check(gpu, box(dims, 15, cap=(0, 1), term=(0, 1), keep=0.5))


@pytest.mark.parametrize("dims", [(30, 30), (10, 9, 12)])
@pytest.mark.parametrize("what", ["parallel arc", "s-t arc", "far arc", "wrap"])
def test_almost_lattices_take_the_list_solver(gpu, dims, what):
    def tweak(tail, head, c, vert, s, t):
        a, b = {"parallel arc": (vert[0], vert[1]), "s-t arc": (s, t), "far arc": (vert[0], vert[-1]),
                "wrap": (vert[dims[-1] - 1], vert[dims[-1]])}[what]
        return np.append(tail, a), np.append(head, b), np.append(c, 7)

    check(gpu, box(dims, 21, tweak=tweak))


@pytest.mark.parametrize("dims", [(70, 90), (18, 20, 22)])
def test_relabel_ratios_and_streams(gpu, dims):
    import torch

    g = box(dims, 31)
    for ratio in (1e-6, 0.5, 50.0):  # a push phase of no time still visits tiles
        check(gpu, g, gr_time_ratio=ratio)
    check(gpu, g, use_graph=1)
    # two graphs on two streams and threads at once
    import threading

    csr = gpu.build_csr(g.n, g.tail, g.head, g.cap)
    ref = oracle.maxflow(g.n, g.s, g.t, g.tail, g.head, g.cap)["value"]
    got = []

    def work():
        dev = torch.device("cuda", 0)
        arrays = [torch.from_numpy(a).to(dev) for a in (csr.row_offsets, csr.head, csr.cap, csr.rev)]
        st = torch.cuda.Stream()
        torch.cuda.synchronize()
        G = gpu.Graph.from_device(g.n, *arrays, g.s, g.t, stream=st)
        v = torch.zeros(1, dtype=torch.int64, device=dev)
        torch.cuda.synchronize()
        for _ in range(5):
            G.solve_device(v, stream=st)
            got.append(int(v.item()))
        G.close()

    th = [threading.Thread(target=work) for _ in range(2)]
    for x in th:
        x.start()
    for x in th:
        x.join()
    assert got == [ref] * 10
