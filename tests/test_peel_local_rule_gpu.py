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


_CHILD = r"""
import sys
import numpy as np
import torch
sys.path.insert(0, sys.argv[1])
import graphgen as gg
import oracle
import paper_2402_15253_gb300 as pico
torch.cuda.set_device(0)
algos = set()
for g in (gg.er_graph(30000, 90000, 1), gg.rmat_graph(14, 12, 2), gg.star_graph(40000),
          gg.grid_graph(60, 70)):
    want = oracle.bz_coreness(*g.numpy())
    for off in (torch.int32, torch.int64):
        got = pico.coreness(g.row_ptr.to("cuda", dtype=off), g.col_idx.cuda(), "auto")
        assert np.array_equal(got.cpu().numpy(), want)
        algos.add(pico.pico_get_stats()["algo"])
print("RESULT", sorted(algos))
"""


@pytest.mark.parametrize("waves", ["0", "1"])
def test_selection_with_and_without_asynchronous_levels(pico, waves):
    """AUTO by either form of PeelOne: PICO_PEEL_WAVES=1 keeps it in the selection's
    own kernel. Both methods are chosen for some graph."""
    import os
    import subprocess
    import sys
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", _CHILD, root], capture_output=True, text=True,
                       env=dict(os.environ, PICO_PEEL_WAVES=waves), timeout=300)
    assert r.returncode == 0, r.stderr
    assert r.stdout.strip().splitlines()[-1] == "RESULT [0, 1]"
