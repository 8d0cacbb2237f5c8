"""Which graphs one CTA peels: all small ones (12,288 vertices, or 20,480 with at
most 400 Ki arcs), and up to 51,200 vertices those whose
degrees are skewed or a lattice's; the grid kernel keeps the others. Either way the
result is the oracle's."""
import numpy as np
import pytest
import torch

import graphgen as gg
import oracle

pytestmark = pytest.mark.gpu

ANY = 20480      # vertices up to which the degrees do not matter


@pytest.fixture(scope="module")
def pico():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2402_15253_gb300 as p
    torch.cuda.set_device(0)
    return p


GRAPHS = [
    ("er-last", lambda: gg.er_graph(ANY, 4 * ANY, 1), True),
    ("er-first", lambda: gg.er_graph(ANY + 1, 4 * ANY, 1), False),
    ("er-few", lambda: gg.er_graph(12288, 300000, 6), True),
    ("er-arcs", lambda: gg.er_graph(12289, 300000, 6), False),
    ("er-51200", lambda: gg.er_graph(51200, 300000, 2), False),
    ("er-sparse", lambda: gg.er_graph(51200, 40000, 3), False),
    ("lattice", lambda: gg.grid_graph(200, 256), True),
    ("chunglu", lambda: gg.chung_lu_graph(30000, 4, clique=60), True),
    ("hub", lambda: gg.star_graph(40000), True),
    ("rmat", lambda: gg.rmat_graph(15, 6, 5), True),
]


@pytest.mark.parametrize("off", [torch.int32, torch.int64], ids=["int32", "int64"])
@pytest.mark.parametrize("name,make,one_cta", GRAPHS, ids=[g[0] for g in GRAPHS])
def test_form(pico, name, make, one_cta, off):
    g = make()
    rp, ci = g.numpy()
    want = oracle.bz_coreness(rp, ci)
    _, ost = oracle.peelone(rp, ci)
    for algo in ("peelone", "auto"):
        got = pico.coreness(g.row_ptr.to("cuda", dtype=off), g.col_idx.cuda(), algo).cpu().numpy()
        st = pico.pico_get_stats()
        assert np.array_equal(got, want)
        if st["algo"] == pico.PICO_ALGO_PEELONE:
            assert (st["blocks"] == 1) == one_cta
            assert st["levels"] == ost["levels"] and st["arcs"] == ost["arcs_scanned"]
            assert st["atomics"] - st["extra"] == ost["decrements"]
        else:
            assert algo == "auto"
