"""What a call's scratch grows by with the graph, as reported without a GPU: one
histogram slot and the chunk entries per arc for HistoCore (and for the method
selection, which may run it), the chunk entries alone for PeelOne."""
import pytest

import paper_2402_15253_gb300 as pico
from paper_2402_15253_gb300 import build as libbuild


@pytest.fixture(scope="module", autouse=True)
def library():
    libbuild.build()


@pytest.mark.parametrize("algo,per_arc", [("histocore", 4.75), ("auto", 4.75), ("peelone", 0.75)])
def test_bytes_per_arc(algo, per_arc):
    a = pico.ALGOS[algo]
    n, m = 1 << 24, 1 << 32
    grown = pico.pico_workspace_bytes(n, 2 * m, a) - pico.pico_workspace_bytes(n, m, a)
    assert grown <= per_arc * m
