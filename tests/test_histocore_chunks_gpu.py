"""HistoCore's compacted chunks (rows of more than 32 arcs, pushed in chunks of
256): chunk lengths around the shortest that is compacted, lists that fill most
of a chunk, estimates that fall below a list's bound (rebuilt), and hubs whose
neighbours mostly lie far below them. Every round must be Alg. 6's."""
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
    yield p
    p.pico_set_histo_update(p.PICO_UPDATE_AUTO, p.PULL_PCT_DEFAULT)


def hub_over(n, core, leaves, seed):
    """A dense core whose members also have `leaves` neighbours of falling
    degree each: their estimates drop over many rounds."""
    gen = torch.Generator().manual_seed(seed)
    i, j = torch.triu_indices(core, core, 1)
    keep = torch.rand(i.numel(), generator=gen) < 0.7
    s, d = [i[keep]], [j[keep]]
    for h in range(core):
        to = core + (torch.rand(leaves, generator=gen) ** 3 * (n - core)).long()
        s.append(torch.full((leaves,), h))
        d.append(to.clamp(max=n - 1))
    return gg.csr_from_pairs(torch.cat(s), torch.cat(d), n)


GRAPHS = [
    # last chunks of 255, 256, 1, 15, 16 and 17 arcs
    ("stars", lambda: gg.disjoint_union([gg.star_graph(k) for k in
                                         (255, 256, 257, 271, 272, 273, 511, 512, 513)])),
    ("hub-33..48", lambda: gg.disjoint_union([gg.star_graph(k) for k in range(31, 50)])),
    ("cliques", lambda: gg.disjoint_union([gg.complete_graph(k) for k in (34, 49, 130, 257, 300)])),
    ("hubs-few", lambda: hub_over(6000, 60, 900, 1)),
    ("hubs-many", lambda: hub_over(9000, 400, 500, 2)),
    ("chain-of-hubs", lambda: gg.chung_lu_graph(1 << 15, 61, clique=150)),
    ("rmat-14", lambda: gg.rmat_graph(14, 20, 62)),
]


@pytest.mark.parametrize("mode", ["push", "auto"])
@pytest.mark.parametrize("off", [torch.int32, torch.int64], ids=["int32", "int64"])
@pytest.mark.parametrize("name,make", GRAPHS, ids=[g[0] for g in GRAPHS])
def test_rounds_match_oracle(pico, name, make, off, mode):
    g = make()
    rp, ci = g.numpy()
    assert pico.pico_set_histo_update(pico.UPDATES[mode], 50) == 0
    got = pico.coreness(g.row_ptr.to("cuda", dtype=off), g.col_idx.cuda(), "histocore").cpu().numpy()
    st = pico.pico_get_stats()
    assert np.array_equal(got, oracle.bz_coreness(rp, ci))
    _, ost = oracle.histocore(rp, ci)
    assert st["rounds"] == ost["rounds"] and st["frontier"] == ost["frontier"]
    assert st["slots"] == ost["slots_read"]
    assert st["arcs"] == g.arcs + ost["arcs_scanned"]
    assert st["atomics"] == g.arcs + 2 * ost["updates"]


def rings_of_hubs(hubs, deg, step):
    """Hubs of `deg` to `deg + step * hubs` neighbours each, joined to each other:
    chunks of which none, a few or all slots lie above the hub's estimate."""
    i, j = torch.triu_indices(hubs, hubs, 1)
    s, d, at = [i], [j], hubs
    for h in range(hubs):
        k = deg + step * h
        leaf = at + torch.arange(k)
        s += [torch.full((k,), h), leaf[:-1], leaf[:-2]]
        d += [leaf, leaf[1:], leaf[2:]]
        at += k
    return gg.csr_from_pairs(torch.cat(s), torch.cat(d), at)


@pytest.mark.parametrize("chunk", [64, 256, 4096])
@pytest.mark.parametrize("deg,step", [(1, 1), (190, 3), (460, 7)], ids=str)
def test_lists_within_the_rows(pico, chunk, deg, step):
    """Every chunk size: lists at the end of chunks that are partly in use."""
    g = rings_of_hubs(60, deg, step)
    rp, ci = g.numpy()
    assert pico.pico_set_histo_update(pico.PICO_UPDATE_PUSH, 50) == 0
    assert pico.pico_set_tuning(32, chunk, 512, 21) == 0
    try:
        for off in (torch.int32, torch.int64):
            got = pico.coreness(g.row_ptr.to("cuda", dtype=off), g.col_idx.cuda(), "histocore")
            st = pico.pico_get_stats()
            assert np.array_equal(got.cpu().numpy(), oracle.bz_coreness(rp, ci))
            _, ost = oracle.histocore(rp, ci)
            assert st["rounds"] == ost["rounds"] and st["frontier"] == ost["frontier"]
            assert st["slots"] == ost["slots_read"]
            assert st["atomics"] == g.arcs + 2 * ost["updates"]
    finally:
        pico.pico_set_tuning(32, 256, 512, 21)
