"""A batch is searched over the settings its kernels read, and over nothing else."""
import pytest
import torch

from paper_2402_15253_gb300 import autotune as at


def test_stages_by_what_is_read():
    assert at.batched_stages("histocore", 100) == at.stages(True)
    for algo in ("peelone", "auto"):
        assert at.batched_stages(algo, at.SHARED_VERTICES) == []
        assert at.batched_stages(algo, at.SHARED_VERTICES + 1) == at.stages(False)


@pytest.mark.gpu
def test_a_batch_that_reads_nothing_keeps_the_setting(tmp_path):
    import graphgen as gg
    import __graft_entry__
    __graft_entry__.build()
    import paper_2402_15253_gb300 as pico
    path = tmp_path / "tuning.json"
    pb = gg.pack_graphs([gg.spec_graph(s) for s in gg.batch_specs(8, 3, nmin=100, nmax=5000)], device="cuda")
    kept = (64, 128, 256, 23)
    try:
        assert pico.pico_set_tuning(*kept) == 0
        best, timings = at.tune_batched(pico, pb.vtx_off, pb.arc_off, pb.row_ptr, pb.col_idx, "peelone",
                                        path=str(path))
        assert best == kept and list(timings) == [kept] and timings[kept] > 0
        assert pico.pico_get_tuning() == kept and not path.exists()
    finally:
        pico.pico_set_tuning(*at.DEFAULT)
