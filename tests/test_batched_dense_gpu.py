"""Batches of graphs with few vertices and many arcs: a graph that holds more arcs than
an SM's share of the batch takes an SM of its own."""
import time

import numpy as np
import pytest
import torch

import graphgen as gg
import oracle

pytestmark = pytest.mark.gpu

TINY_ARCS = 32 << 10


@pytest.fixture(scope="module")
def pico():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2402_15253_gb300 as p
    torch.cuda.set_device(0)
    return p


def solve(pico, graphs):
    pb = gg.pack_graphs(graphs, device="cuda")
    tv, ta = int(pb.vtx_off[-1]), int(pb.arc_off[-1])
    out = torch.empty(tv, dtype=torch.int32, device="cuda")

    def call():
        assert pico.pico_coreness_batched(pb.vtx_off, pb.arc_off, pb.G, pb.row_ptr, pb.col_idx, tv,
                                          ta, out, pico.PICO_ALGO_PEELONE) == pico.PICO_OK
    return call, out


BATCHES = [
    # one dense graph; as many as an SM's share allows; around the least arcs; with others
    ("one", lambda: [gg.er_graph(2000, 300000, 1)]),
    ("complete", lambda: [gg.complete_graph(k) for k in (180, 181, 182, 183, 2048)]),
    ("least", lambda: [gg.er_graph(300, TINY_ARCS // 2 + k, 2) for k in (-1, 0, 1, 400)]),
    ("many", lambda: [gg.er_graph(500 + i, 30000, i) for i in range(200)]),
    ("among", lambda: [gg.er_graph(2048, 400000, 3), gg.er_graph(2049, 400000, 4), gg.star_graph(9),
                       gg.rmat_graph(11, 200, 5), gg.er_graph(60000, 90000, 6), gg.grid_graph(20, 30)]),
]


@pytest.mark.parametrize("name,make", BATCHES, ids=[b[0] for b in BATCHES])
def test_dense_batches(pico, name, make):
    graphs = make()
    call, out = solve(pico, graphs)
    call()
    want = np.concatenate([oracle.bz_coreness(*g.numpy()) for g in graphs])
    assert np.array_equal(out.cpu().numpy(), want)
    st = pico.pico_get_stats()
    assert st["arcs"] == sum(g.arcs for g in graphs) and st["kmax"] == int(want.max())
    assert st["atomics"] - st["extra"] == st["arcs"] - int(want.sum())


def test_dense_graph_is_not_held_to_few_threads(pico):
    """The same 16 graphs with 2,000 vertices and with 49 isolated ones more, which
    makes them large enough for an SM each by their vertices (128 threads took 3.7 times
    as long)."""
    g = gg.er_graph(2000, 400000, 7)
    more = gg.disjoint_union([g, gg.from_edge_list([], 49)])
    best = {}
    for name, graph in (("few", g), ("more", more)):
        call, _ = solve(pico, [graph] * 16)
        for _ in range(8):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            call()
            torch.cuda.synchronize()
            best[name] = min(best.get(name, 1.0), time.perf_counter() - t0)
    assert best["few"] < 1.5 * best["more"]
