"""PeelOne's light levels on one cluster, between launches of the grid kernel.

Every graph here is handed over, which the phase counts show: "wave_mid" counts
the launches that peeled on the cluster, "init" the initialisation and every wave
that the grid kernel took back. Results and counts of work are the
oracle's.
"""
import numpy as np
import pytest
import torch

import graphgen as gg
import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pico():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2402_15253_gb300 as p
    torch.cuda.set_device(0)
    return p


def peel(pico, g, off):
    """Compares with the oracle; returns (cluster launches, waves taken back)."""
    rp, ci = g.numpy()
    want = oracle.bz_coreness(rp, ci)
    _, ost = oracle.peelone(rp, ci)
    got = pico.coreness(g.row_ptr.to("cuda", dtype=off), g.col_idx.cuda(), "peelone").cpu().numpy()
    st = pico.pico_get_stats()
    assert np.array_equal(got, want), f"{int((got != want).sum())} vertices differ"
    assert st["levels"] == ost["levels"] and st["kmax"] == ost["kmax"]
    assert st["arcs"] == ost["arcs_scanned"]
    assert st["atomics"] - st["extra"] == ost["decrements"]
    ph = st["phases"]
    return ph.get("wave_mid", {"count": 0})["count"], ph["init"]["count"] - 1


def circulant(n, reach, first=0):
    """Pairs of n vertices from `first` on, each joined to the next `reach`."""
    i = torch.arange(n, dtype=torch.int64).repeat_interleave(reach)
    d = torch.arange(1, reach + 1, dtype=torch.int64).repeat(n)
    return first + i, first + (i + d) % n


def union(n, *pairs):
    return gg.csr_from_pairs(torch.cat([p[0] for p in pairs]), torch.cat([p[1] for p in pairs]), n)


def star(hub, ends):
    return torch.full_like(ends, hub), ends


def strips(count):
    """`count` strips of 500 squares of distinct widths over one dense part: each
    peels from its end in waves of a few vertices, many in a row."""
    core = 60000
    pairs = [circulant(core, 24), star(0, torch.arange(30, 6000))]
    at = core
    for c in range(count):
        w = 4 + c
        ids = at + torch.arange(500 * w, dtype=torch.int64).view(500, w)
        pairs.append((ids[:-1].reshape(-1), ids[1:].reshape(-1)))
        # each vertex is held by w others of its strip's next column
        for s in range(1, w):
            pairs.append((ids[:-1].reshape(-1), ids[1:].roll(s, 1).reshape(-1)))
        pairs.append((ids[-1].repeat_interleave(30), torch.arange(30).repeat(w) + 100 * c))
        at += 500 * w
    return union(at, *pairs)


def near_overflow():
    """More residual vertices inside the first window than the near lists hold."""
    n = 300000
    gen = torch.Generator().manual_seed(7)
    return union(n, (torch.randint(n, (10 * n,), generator=gen), torch.randint(n, (10 * n,), generator=gen)),
                 star(5, torch.arange(6, 9000)))


@pytest.mark.parametrize("off", [torch.int32, torch.int64], ids=["int32", "int64"])
@pytest.mark.parametrize("make", [lambda: strips(20), near_overflow], ids=["strips", "near-overflow"])
def test_consecutive_waves(pico, make, off):
    g = make()
    for _ in range(3):
        launches, _ = peel(pico, g, off)
        assert launches >= 1


def test_error_of_a_handed_over_call_is_reported(pico):
    """A launch of which only some CTAs finish does not keep the narrower one
    after it from publishing the error."""
    assert pico.pico_selftest_handover() == pico.PICO_ERR_TIMEOUT
    assert pico.pico_last_device_status() == pico.PICO_OK


def hub_in_wide_wave(core, leaves):
    """A wave of 600 vertices at level 2, one of them with `leaves` neighbours that
    left at level 1: more arcs than the cluster kernel may walk."""
    a = core + torch.arange(300)
    b = core + 300 + torch.arange(600)
    leaf = core + 900 + torch.arange(leaves)
    return union(core + 900 + leaves, circulant(core, 12), star(0, torch.arange(20, 8000)),
                 (a.repeat_interleave(2), b), (b, torch.arange(600) * 7 + 1),
                 (b, torch.arange(600) * 7 + 9001), star(int(b[77]), leaf))


def five_tree(core):
    """A tree of five children a vertex, whose 78,125 leaves hang on a dense part:
    level 5 peels it from the root, and its last waves do not fit the queues."""
    size = [5 ** i for i in range(8)]
    first = [core + sum(size[:i]) for i in range(8)]
    pairs = [circulant(core, 12), star(0, torch.arange(20, 6000))]
    for i in range(1, 8):
        ids = torch.arange(size[i])
        pairs.append((first[i - 1] + ids // 5, first[i] + ids))
    leaf = first[7] + torch.arange(size[7])
    for j in range(5):
        pairs.append((leaf, (torch.arange(size[7]) * 31 + j * 7001) % core))
    return union(first[7] + size[7], *pairs)


def alternating(parts, first, step):
    """Heavy levels (9,000 vertices of a complete bipartite part each) with light
    ones between them, next to a star."""
    graphs = [gg.star_graph(90000)]
    for i in range(parts):
        k = first + step * i
        left = torch.arange(k).repeat_interleave(9000)
        graphs += [gg.csr_from_pairs(left, k + torch.arange(9000).repeat(k), k + 9000),
                   gg.complete_graph(k + 6)]
    return gg.disjoint_union(graphs)


TURNS = [
    # (graph, launches that peel on the cluster, waves the grid kernel takes back)
    ("wide-wave-with-hub", lambda: hub_in_wide_wave(300000, 200000), None, 1),
    ("wide-wave-with-hub-last", lambda: hub_in_wide_wave(70000, 200000), 1, 0),
    ("spilled-last", lambda: five_tree(60000), 1, 0),
    ("spilled-back", lambda: five_tree(300000), None, 1),
    # one launch below 6 Mi arcs, on the cluster; four below 20 Mi (the second of the
    # cluster walks these heavy levels), then six: the last on the grid
    ("turns-end-on-the-cluster", lambda: alternating(5, 15, 8), 1, 0),
    ("four-turns", lambda: alternating(7, 37, 13), 2, 1),
    ("turns-end-on-the-grid", lambda: alternating(10, 37, 25), 3, 3),
    ("late-budget", lambda: alternating(3, 37, 80), 2, 2),
]


@pytest.mark.parametrize("off", [torch.int32, torch.int64], ids=["int32", "int64"])
@pytest.mark.parametrize("name,make,clusters,back", TURNS, ids=[t[0] for t in TURNS])
def test_turns(pico, name, make, clusters, back, off):
    launches, taken_back = peel(pico, make(), off)
    assert launches == clusters if clusters is not None else launches >= 1
    assert taken_back >= back if clusters is None else taken_back == back
