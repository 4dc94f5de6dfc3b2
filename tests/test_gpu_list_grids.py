"""The list solver on single 2D and 3D grids with default options, which the lattice solvers take over: one more arc
beside another keeps a grid off them. CTA-local lists and BFS hops, cut-only solves, and the build with checked
gathers; and graphs that are almost lattices run the list solver, lattices the lattice solvers."""
import numpy as np
import pytest

import oracle
from paper_1507_01926_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def extra(g, tail, head):
    """g with one more arc (capacity 7)."""
    return I.Instance(g.n, g.s, g.t, np.append(g.tail, tail).astype(np.int32), np.append(g.head, head).astype(np.int32),
                      np.append(g.cap, 7).astype(np.int32), g.name)


def arc(g, what):
    inner = np.flatnonzero((g.tail != g.s) & (g.head != g.t) & (g.tail != g.t) & (g.head != g.s))[0]
    width = {"grid2d": 80, "grid3d": 40}[g.name[:6]]  # cells in a row of GRIDS
    return {"wrap": (width - 1, width), "parallel arc": (g.tail[inner], g.head[inner]), "s-t arc": (g.s, g.t), "far arc": (0, g.n - 3)}[what]


def solve_and_check(mf, g, lattice, **opts):
    csr = mf.build_csr(g.n, g.tail, g.head, g.cap)
    ref = oracle.maxflow(g.n, g.s, g.t, g.tail, g.head, g.cap, want_flow=False)
    with mf.Graph.from_csr(csr, g.s, g.t, mf.default_options(**opts)) as G:
        for _ in range(2):
            r = G.solve(flow=not opts.get("cut_only"))
            assert any(G.stats()["rounds_by_size"]) != lattice, g.name
            cut = mf.cut_bits_to_bool(r.cut_bits, g.n)
            assert r.value == ref["value"] and np.array_equal(cut, ref["cut"]), g.name
            if r.flow is not None:
                f = np.where(csr.arc_slot >= 0, r.flow[np.maximum(csr.arc_slot, 0)], 0).astype(np.int64)
                assert not oracle.check_flow(g.n, g.s, g.t, g.tail, g.head, g.cap, f, r.value, cut), g.name


GRIDS = {"2d": lambda: I.grid2d(96, 80, 91), "3d": lambda: I.grid3d(40, 36, 28, 92)}


@pytest.mark.parametrize("opts", [{}, dict(bfs_hops=1), dict(bfs_hops=64), dict(cut_only=1), dict(use_graph=1)])
@pytest.mark.parametrize("which", sorted(GRIDS))
def test_default_lists_on_grids(gpu, which, opts):
    g = GRIDS[which]()
    solve_and_check(gpu, extra(g, *arc(g, "parallel arc")), False, **opts)


@pytest.mark.parametrize("what", ["parallel arc", "s-t arc", "far arc", "wrap"])
@pytest.mark.parametrize("which", sorted(GRIDS))
def test_almost_lattices_run_the_list_solver(gpu, which, what):
    g = GRIDS[which]()
    solve_and_check(gpu, g, True)
    solve_and_check(gpu, extra(g, *arc(g, what)), False)


@pytest.mark.parametrize("opts", [{}, dict(cut_only=1), dict(bin_thread=2, bin_warp=4)])
@pytest.mark.parametrize("make", [lambda: I.grid2d(40, 37, 1), lambda: I.grid3d(20, 18, 12, 2)], ids=["2d", "3d"])
def test_checked_lists_on_grids(gpu, make, opts):
    from paper_1507_01926_gb300 import build as mfbuild

    g = make()
    before = gpu.use_library(mfbuild.build(check=True))
    try:
        solve_and_check(gpu, extra(g, *arc(g, "parallel arc")), False, **opts)
    finally:
        gpu.use_library(before)
