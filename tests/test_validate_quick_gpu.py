"""Validation of a graph in even shares of its arcs: rows that begin and end
around a share (512 arcs), runs of empty rows, hubs, and single defects
anywhere must be judged as by a plain check of every arc."""
import time

import numpy as np
import pytest
import torch

import graphgen as gg

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pico():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2402_15253_gb300 as p
    torch.cuda.set_device(0)
    return p


def defects(pico, rp, ci):
    """Every arc looked at, in numpy. An id outside [0, n) is reported as such
    and compared with nothing."""
    n = len(rp) - 1
    row = np.repeat(np.arange(n), np.diff(rp))
    bits = 0
    ok = (ci >= 0) & (ci < n)
    if not ok.all():
        bits |= pico.PICO_DEFECT_IDS
    if (ci == row).any():
        bits |= pico.PICO_DEFECT_LOOP
    same = row[1:] == row[:-1]
    if (same & ok[:-1] & (ci[1:] <= ci[:-1])).any():
        bits |= pico.PICO_DEFECT_ORDER
    arcs = set(zip(row[ok].tolist(), ci[ok].tolist()))
    if any((u, v) not in arcs for v, u in arcs):
        bits |= pico.PICO_DEFECT_ASYMMETRIC
    return bits


def spread(parts, gap):
    """The parts' union with `gap` isolated vertices before, between and after."""
    out = [gg.from_edge_list([], gap)] if gap else []
    for p in parts:
        out += [p] + ([gg.from_edge_list([], gap)] if gap else [])
    return gg.disjoint_union(out)


GRAPHS = [
    ("cliques", lambda: spread([gg.complete_graph(k) for k in (2, 17, 23, 24, 33)], 0)),
    ("gaps-1", lambda: spread([gg.complete_graph(5)] * 40, 1)),
    ("gaps-31", lambda: spread([gg.complete_graph(6)] * 30, 31)),
    ("gaps-32", lambda: spread([gg.path_graph(3)] * 30, 32)),
    ("gaps-700", lambda: spread([gg.star_graph(511), gg.star_graph(512), gg.star_graph(513)], 700)),
    ("hub", lambda: gg.star_graph(5000)),
    ("rmat", lambda: gg.rmat_graph(11, 8, 5)),
    ("single-arc-rows", lambda: spread([gg.complete_graph(2)] * 700, 0)),
]


@pytest.mark.parametrize("off", [torch.int32, torch.int64], ids=["int32", "int64"])
@pytest.mark.parametrize("name,make", GRAPHS, ids=[g[0] for g in GRAPHS])
def test_shares_of_arcs(pico, name, make, off):
    g = make()
    rp, ci = g.numpy()
    n, m = g.n, len(ci)
    check = pico.pico_validate_graph if off == torch.int32 else pico.pico_validate_graph_i64
    drp = torch.from_numpy(rp).to("cuda", dtype=off)
    assert check(drp, torch.from_numpy(ci).cuda(), n, m) == (pico.PICO_OK, 0)
    rng = np.random.default_rng(3)
    places = {0, m - 1, m // 2} | {p for p in (511, 512, 513) if p < m}
    for at in sorted(places):
        for value in (n, -1, int(rng.integers(n)), int(np.searchsorted(rp, at, "right") - 1)):
            bad = ci.copy()
            bad[at] = value
            want = defects(pico, rp, bad)
            status, bits = check(drp, torch.from_numpy(bad).cuda(), n, m)
            if want & pico.PICO_DEFECT_ORDER:   # an unsorted row may hide an arc or seem to
                mask = ~pico.PICO_DEFECT_ASYMMETRIC
                assert bits & mask == want & mask, (at, value)
            else:
                assert bits == want, (at, value)
            assert (status == pico.PICO_OK) == (bits == 0)


@pytest.mark.parametrize("off", [torch.int32, torch.int64], ids=["int32", "int64"])
@pytest.mark.parametrize("gap", [31, 32, 33, 63, 64, 65, 95, 96, 97, 1023, 1024, 1025, 1 << 20])
def test_runs_of_empty_rows(pico, gap, off):
    """Used ids with runs of unused ones between them, inside one share of arcs."""
    g = spread([gg.complete_graph(3), gg.path_graph(2), gg.complete_graph(4)] * 2, gap)
    rp, ci = g.numpy()
    check = pico.pico_validate_graph if off == torch.int32 else pico.pico_validate_graph_i64
    drp = torch.from_numpy(rp).to("cuda", dtype=off)
    assert check(drp, torch.from_numpy(ci).cuda(), g.n, len(ci)) == (pico.PICO_OK, 0)
    for at in range(len(ci)):
        bad = ci.copy()
        bad[at] = ci[at - 1]
        want = defects(pico, rp, bad)
        status, bits = check(drp, torch.from_numpy(bad).cuda(), g.n, len(ci))
        assert bits & ~pico.PICO_DEFECT_ASYMMETRIC == want & ~pico.PICO_DEFECT_ASYMMETRIC, at
        assert (status == pico.PICO_OK) == (want == 0), at


def test_long_run_of_empty_rows_is_not_walked(pico):
    """2^23 unused ids between two used ranges: some 20 dependent steps, not a
    quarter of a million (95 ms)."""
    g = spread([gg.complete_graph(5)] * 2, 1 << 23)
    rp, ci = g.row_ptr.cuda(), g.col_idx.cuda()
    times = []
    for _ in range(4):
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        assert pico.pico_validate_graph(rp, ci, g.n, g.arcs) == (pico.PICO_OK, 0)
        times.append(time.perf_counter() - t0)
    assert min(times) < 0.02


def test_malformed_graph_costs_little_more(pico):
    """One bad id among 2,000 rows of 200 arcs: the exact kernel that names the
    defect has a warp for every row (a 32nd of them took seven times as long)."""
    g = gg.er_graph(2000, 200000, 9)
    rp, ci = g.row_ptr.cuda(), g.col_idx.cuda()
    bad = ci.clone()
    bad[g.arcs // 2] = g.n
    best = {}
    for name, c, want in (("valid", ci, 0), ("bad", bad, pico.PICO_DEFECT_IDS)) * 8:
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        assert pico.pico_validate_graph(rp, c, g.n, g.arcs)[1] & want == want
        best[name] = min(best.get(name, 1.0), time.perf_counter() - t0)
    assert best["bad"] < 3 * best["valid"]
