"""Counters of the grid-wide phase: its launches number a run's waves in one
sequence.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)
    from paper_1507_01490_gb300 import _build, bcm
    _build.build_cuda()
    bcm.load()
    return bcm


def test_trace_numbers_a_runs_waves(B, gen):
    several = 0
    for g in (gen.ba(40000, 3, seed=8), gen.rmat(15, 6, seed=10), gen.chung_lu(60000, 8.0, 2.3, seed=2)):
        with B.BcmGraph.from_graph(g) as h:
            for k in (10, 100):
                st = h.topk(k, flags=B.BCM_TRACE, heavy_words=1)[3]
                rec, count = h.trace()
                assert count == len(rec)
                kind = (rec[:, 1] >> np.uint64(60)).astype(int)
                wave = ((rec[:, 1] >> np.uint64(32)) & np.uint64(0xfffffff)).astype(int)
                level = (rec[:, 1] & np.uint64(0xffffffff)).astype(int)
                ends = wave[kind == B.TRACE_GRID_WAVE]
                assert sorted(ends.tolist()) == list(range(st["grid_waves"])), (g.name, k)
                starts = list(zip(wave[kind == B.TRACE_GRID_LEVEL].tolist(), level[kind == B.TRACE_GRID_LEVEL].tolist()))
                assert len(set(starts)) == len(starts) == st["grid_levels"], (g.name, k)
                several += st["grid_waves"] > 2
    assert several   # (the first wave or two, and those of the launches behind the prefilter)
