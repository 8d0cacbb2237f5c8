"""The forms of PeelOne, at the sizes where each begins and ends.

A single graph is peeled in one CTA's shared memory (small), by the grid
kernel, or by the grid kernel and the cluster kernel in turn (skewed graphs);
a batched graph in a CTA's or a cluster's shared memory, or in a cluster's
global memory. Every form must return the oracle's coreness and count its
levels, arcs and decrements, which do not depend on the order of a level.
"""
import numpy as np
import pytest
import torch

import graphgen as gg
import oracle

pytestmark = pytest.mark.gpu

SLOTS = 51200          # residual degrees of one CTA
LOCAL_ARCS = 640 << 10  # arcs up to which a single graph takes one CTA
CLUSTER_SLOTS = 4 * SLOTS
TINY = 2048


@pytest.fixture(scope="module")
def pico():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2402_15253_gb300 as p
    torch.cuda.set_device(0)
    return p


def check_single(pico, g, off, algos=("peelone",)):
    rp, ci = g.numpy()
    want = oracle.bz_coreness(rp, ci)
    _, ost = oracle.peelone(rp, ci)
    drp, dci = g.row_ptr.to("cuda", dtype=off), g.col_idx.cuda()
    for algo in algos:
        got = pico.coreness(drp, dci, algo).cpu().numpy()
        st = pico.pico_get_stats()
        assert np.array_equal(got, want), f"{int((got != want).sum())} vertices differ ({algo})"
        if st["algo"] == pico.PICO_ALGO_PEELONE:
            assert st["levels"] == ost["levels"] and st["kmax"] == ost["kmax"]
            assert st["arcs"] == ost["arcs_scanned"]
            assert st["atomics"] - st["extra"] == ost["decrements"]


def ring_of(n, extra_every=0):
    """A cycle on n vertices, every extra_every-th vertex joined to the next but one."""
    i = torch.arange(n, dtype=torch.int64)
    s, d = [i], [(i + 1) % n]
    if extra_every:
        j = i[::extra_every]
        s.append(j)
        d.append((j + 2) % n)
    return gg.csr_from_pairs(torch.cat(s), torch.cat(d), n)


def bipartite(a, b):
    s = torch.arange(a).repeat_interleave(b)
    d = a + torch.arange(b).repeat(a)
    return gg.csr_from_pairs(s, d, a + b)


def nested_hubs(n, hubs, seed):
    """Hubs of widely different degrees over a sparse random graph: many levels
    of few vertices with long rows."""
    gen = torch.Generator().manual_seed(seed)
    s = [torch.randint(n, (2 * n,), generator=gen)]
    d = [torch.randint(n, (2 * n,), generator=gen)]
    for h in range(hubs):
        deg = 40 + 37 * h
        s.append(torch.full((deg,), h))
        d.append(torch.randint(hubs, (deg,), generator=gen) if h % 2 else
                 torch.randint(n, (deg,), generator=gen))
    i, j = torch.triu_indices(hubs, hubs, 1)
    keep = torch.rand(i.numel(), generator=gen) < 0.5
    s.append(i[keep])
    d.append(j[keep])
    return gg.csr_from_pairs(torch.cat(s), torch.cat(d), n)


SINGLE = [
    # the last size of the shared-memory form and the first beyond it
    ("slots", lambda: ring_of(SLOTS, 3)),
    ("slots+1", lambda: ring_of(SLOTS + 1, 3)),
    ("arcs", lambda: bipartite(64, LOCAL_ARCS // 128)),
    ("arcs+", lambda: bipartite(64, LOCAL_ARCS // 128 + 1)),
    # rows around a piece (128, 256 arcs) and more pieces than are listed at once
    ("rows-127..257", lambda: gg.disjoint_union([gg.complete_graph(k) for k in
                                                 (2, 33, 128, 129, 130, 256, 257, 258)])),
    ("star-51199", lambda: gg.star_graph(SLOTS - 1)),
    ("narrow-2048", lambda: ring_of(2048, 2)),
    ("narrow+1", lambda: ring_of(2049, 2)),
    ("one-edge", lambda: gg.from_edge_list([(3, 1)], 5)),
    # handed over to the cluster kernel: a queue beyond a CTA's share of a level,
    # rows longer than a segment, a residual list beyond the near window
    ("hubs-60k", lambda: nested_hubs(60000, 400, 1)),
    ("hubs-300k", lambda: nested_hubs(300001, 900, 2)),
    ("chunglu-2^18", lambda: gg.chung_lu_graph(1 << 18, 71, clique=700)),
    ("rmat-17", lambda: gg.rmat_graph(17, 12, 72)),
    # one wide level next to a hub: handed over by its skew, handed back by its size
    ("star-of-rings", lambda: gg.csr_from_pairs(
        torch.cat([torch.arange(200000), torch.zeros(60000, dtype=torch.int64)]),
        torch.cat([(torch.arange(200000) + 1) % 200000, torch.arange(60000) * 3 + 2]), 200000)),
]


@pytest.mark.parametrize("off", [torch.int32, torch.int64], ids=["int32", "int64"])
@pytest.mark.parametrize("name,make", SINGLE, ids=[c[0] for c in SINGLE])
def test_single_graph_forms(pico, name, make, off):
    check_single(pico, make(), off, ("peelone", "auto"))


def test_turns_run_out(pico):
    """More alternations of light and heavy levels than launches: the last
    launch of the grid kernel finishes the run."""
    parts = [gg.rmat_graph(12, 8 + 6 * i, 80 + i) for i in range(8)]
    parts += [bipartite(12 + 25 * i, 9000) for i in range(6)] + [gg.star_graph(90000)]
    check_single(pico, gg.disjoint_union(parts), torch.int32, ("peelone", "auto"))


BATCH = [
    ("tiny", [1, 2, 127, 128, 129, TINY - 1, TINY, TINY + 1]),
    ("middle", [TINY + 1, 4096, 4097, SLOTS - 1, SLOTS]),
    ("large", [SLOTS + 1, 2 * SLOTS + 2, CLUSTER_SLOTS - 3, CLUSTER_SLOTS]),
    ("global", [CLUSTER_SLOTS + 1, 70, SLOTS + 7]),
    ("mixed", [0, 5, 300000, SLOTS, 0, 3000, 60001, TINY]),
]


@pytest.mark.parametrize("name,sizes", BATCH, ids=[c[0] for c in BATCH])
def test_batched_forms(pico, name, sizes):
    graphs = []
    for i, n in enumerate(sizes):
        if n < 3:
            graphs.append(gg.from_edge_list([(0, 1)] if n == 2 else [], n))
        elif i % 3 == 0:
            graphs.append(gg.er_graph(n, 5 * n, 90 + i))
        elif i % 3 == 1:
            graphs.append(gg.spec_graph(gg.BatchSpec("rmat", n, 8.0, 90 + i)))
        else:
            graphs.append(ring_of(n, 5))
    pb = gg.pack_graphs(graphs)
    want = oracle.bz_coreness_batched(pb.vtx_off, pb.arc_off, pb.row_ptr, pb.col_idx)
    d = [t.cuda() for t in (pb.vtx_off, pb.arc_off, pb.row_ptr, pb.col_idx)]
    got = pico.coreness_batched(*d, "peelone").cpu().numpy()
    assert np.array_equal(got, want), f"{int((got != want).sum())} vertices differ"
    st = pico.pico_get_stats()
    assert st["kmax"] == int(want.max())
    assert st["arcs"] == int(pb.arc_off[-1])
    assert st["atomics"] - st["extra"] == int(pb.arc_off[-1]) - int(want.sum())


def test_batched_forms_replayed(pico):
    """Graphs of every size class recorded in one CUDA graph, where the launch
    for the largest runs beside the next one; every replay gives the oracle's
    coreness."""
    graphs = [gg.er_graph(CLUSTER_SLOTS + 9, 900000, 95), ring_of(300000, 5), gg.star_graph(90000),
              gg.er_graph(30000, 120000, 96), gg.complete_graph(60)]
    pb = gg.pack_graphs(graphs)
    want = oracle.bz_coreness_batched(pb.vtx_off, pb.arc_off, pb.row_ptr, pb.col_idx)
    tv, ta = int(pb.vtx_off[-1]), int(pb.arc_off[-1])
    d = [t.cuda() for t in (pb.vtx_off, pb.arc_off, pb.row_ptr, pb.col_idx)]
    out = torch.full((tv,), -1, dtype=torch.int32, device="cuda")
    s, graph = torch.cuda.Stream(), torch.cuda.CUDAGraph()

    def call():
        return pico.pico_coreness_batched(d[0], d[1], len(graphs), d[2], d[3], tv, ta, out,
                                          pico.ALGOS["peelone"], s)

    s.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(s):
        assert call() == pico.PICO_OK
        s.synchronize()
        with torch.cuda.graph(graph, stream=s):
            assert call() == pico.PICO_OK
    for _ in range(2):
        torch.cuda.synchronize()
        out.fill_(-1)
        graph.replay()
        torch.cuda.synchronize()
        assert pico.pico_last_device_status() == pico.PICO_OK
        assert np.array_equal(out.cpu().numpy(), want)
