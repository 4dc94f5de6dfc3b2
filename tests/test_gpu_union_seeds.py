"""Seeds of a union's BFS with more arcs than a CTA has threads are expanded in runs of 1024 arcs by all CTAs instead
of being queued. Terminal degrees at the edges of the thread count and of a run, one and several instances, and a union
whose lists cannot hold the runs (few vertices with very many arcs), where every seed is queued."""
import numpy as np
import pytest

import oracle
from paper_1507_01926_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def star(k, seed, parallel=1):
    """s -> k middle vertices -> t, each arc `parallel` times, and arcs between neighbouring middle vertices."""
    rng = np.random.default_rng(seed)
    mid = np.arange(k)
    tail = np.concatenate([np.repeat(np.full(k, k), parallel), np.repeat(mid, parallel), mid[:-1]])
    head = np.concatenate([np.repeat(mid, parallel), np.repeat(np.full(k, k + 1), parallel), mid[1:]])
    cap = rng.integers(0, 50, tail.size)
    return I.Instance(k + 2, k, k + 1, tail.astype(np.int32), head.astype(np.int32), cap.astype(np.int32), f"star_{k}")


@pytest.mark.parametrize("sizes,parallel", [((255,), 1), ((256, 257), 1), ((1023, 1024, 1025), 1), ((3000, 5, 64), 1),
                                            ((3, 4), 3000)])
@pytest.mark.parametrize("opts", [{}, dict(block_threads=64), dict(instance_relabel=0), dict(cut_only=1),
                                  dict(simple_rounds=1)])
def test_union_terminals(gpu, sizes, parallel, opts):
    insts = [star(k, 70 + k, parallel) for k in sizes]
    csrs = [gpu.build_csr(g.n, g.tail, g.head, g.cap) for g in insts]
    with gpu.Batch(csrs, [(g.s, g.t) for g in insts], gpu.default_options(**opts)) as B:
        res = B.solve(flow=not opts.get("cut_only"))
    for g, c, r in zip(insts, csrs, res):
        ref = oracle.maxflow(g.n, g.s, g.t, g.tail, g.head, g.cap, want_flow=False)
        cut = gpu.cut_bits_to_bool(r.cut_bits, g.n)
        assert r.value == ref["value"] and np.array_equal(cut, ref["cut"]), g.name
        if not opts.get("cut_only"):
            f = np.where(c.arc_slot >= 0, r.flow[np.maximum(c.arc_slot, 0)], 0).astype(np.int64)
            assert not oracle.check_flow(g.n, g.s, g.t, g.tail, g.head, g.cap, f, r.value, cut), g.name


def test_service_requests(gpu):
    insts = [star(k, 80 + k) for k in (127, 128, 129, 2049)] + [I.grid2d(60, 50, 81)]
    csrs = [gpu.build_csr(g.n, g.tail, g.head, g.cap) for g in insts]
    with gpu.Service(1 << 30) as svc:
        tickets = [svc.submit(c, g.s, g.t) for c, g in zip(csrs, insts)]
        for k, g in zip(tickets, insts):
            assert svc.wait(k, 120000) is not None
            r = svc.poll(k)
            ref = oracle.maxflow(g.n, g.s, g.t, g.tail, g.head, g.cap, want_flow=False)
            assert r.value == ref["value"] and np.array_equal(gpu.cut_bits_to_bool(r.cut_bits, g.n), ref["cut"]), g.name
