"""Vertices with very many arcs: BFS levels cut the arcs of vertices with more than 16384 of them into runs of 1024 that
all CTAs share, and a CTA-wide discharge loads the next chunk of arcs while it works on one. Degrees at the edges of
that bound, of a run and of a chunk, one and several hubs in a level, and a graph whose lists cannot hold the runs (few
vertices with very many arcs), where the CTA that finds a hub walks its arcs."""
import numpy as np
import pytest

import oracle
from paper_1507_01926_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def hubs(degrees, seed, leaves=0):
    """s -> hubs -> leaves -> sink hub -> t; hub i has degrees[i] arcs, the one from s and the others to leaves
    (in order when the leaves are as many, else drawn with repetition), and one to the next hub; every 7th leaf also
    sends to the next one."""
    rng = np.random.default_rng(seed)
    k = leaves or max(degrees) - 1
    leaf = np.arange(k)
    h = k + np.arange(len(degrees))
    back, s, t = k + len(degrees), k + len(degrees) + 1, k + len(degrees) + 2
    tail, head = [np.full(h.size, s), leaf, [back], leaf[:-1:7]], [h, np.full(k, back), [t], leaf[1::7]]
    for v, d in zip(h, degrees):
        tail.append(np.full(d - 1, v))
        head.append(leaf if d - 1 == k else rng.integers(0, k, d - 1))
    if len(degrees) > 1:
        tail.append(h[:-1]), head.append(h[1:])
    size = [len(x) for x in tail]
    cap = [rng.integers(5000, 20000, size[0]), rng.integers(0, 9, size[1]), [3 * k], rng.integers(0, 9, size[3])]
    cap += [rng.integers(0, 9, x) for x in size[4:]]
    tail, head, cap = (np.concatenate(x).astype(np.int32) for x in (tail, head, cap))
    return I.Instance(t + 1, s, t, tail, head, cap, f"hubs_{degrees}")


CASES = {
    "run_minus": lambda: hubs((16384,), 31),
    "run": lambda: hubs((16385,), 32),
    "runs": lambda: hubs((17407, 17407, 20000), 33),
    "chunks": lambda: hubs((256, 257, 1023, 1024, 1025, 2048, 2049), 34),
    "no_room": lambda: hubs((40000, 33000), 35, leaves=40),
}
OPTS = [{}, dict(cut_only=1), dict(simple_rounds=1), dict(bfs_pull=1 << 20), dict(block_threads=64, bin_warp=40)]


@pytest.mark.parametrize("opts", OPTS)
@pytest.mark.parametrize("name", sorted(CASES))
def test_solve_exact(gpu, name, opts):
    g = CASES[name]()
    csr = gpu.build_csr(g.n, g.tail, g.head, g.cap)
    ref = oracle.maxflow(g.n, g.s, g.t, g.tail, g.head, g.cap, want_flow=False)
    with gpu.Graph.from_csr(csr, g.s, g.t, gpu.default_options(**opts)) as G:
        r = G.solve(flow=not opts.get("cut_only"))
    cut = gpu.cut_bits_to_bool(r.cut_bits, g.n)
    assert r.value == ref["value"] and np.array_equal(cut, ref["cut"])
    if not opts.get("cut_only"):
        f = np.where(csr.arc_slot >= 0, r.flow[np.maximum(csr.arc_slot, 0)], 0).astype(np.int64)
        assert not oracle.check_flow(g.n, g.s, g.t, g.tail, g.head, g.cap, f, r.value, cut)


@pytest.mark.parametrize("rounds", [0, 1, 4])
@pytest.mark.parametrize("name", sorted(CASES))
def test_relabel_labels_exact(gpu, name, rounds):
    g = CASES[name]()
    csr = gpu.build_csr(g.n, g.tail, g.head, g.cap)
    with gpu.Graph.from_csr(csr, g.s, g.t) as G:
        res, lab, ex, done = G.run_rounds(rounds, final_relabel=True)
    k = res > 0
    assert np.array_equal(lab, oracle.sink_distances(g.n, g.s, g.t, csr.tails()[k], csr.head[k]))
