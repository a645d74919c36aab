"""Counters of the grid-wide phase: its launches number a run's waves in one
sequence, and a source that the wave picker stops at level 0 scans no arc.
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


def _matchings(rng, n, d):
    return np.concatenate([rng.permutation(n).reshape(-1, 2) for _ in range(d)])


def test_picked_sources_stopped_at_level_0(B, gen, orc):
    """128 stars set a weak threshold in the first wave; six trees of two levels, next by degree, a strong one in the
    second; every vertex of 100 parts of 1,200 (degree about 40) passes the prefilter and is stopped at level 0 when
    the third is picked.  Without those, no more arcs can be scanned than complete searches of the other sources."""
    rng = np.random.default_rng(3)
    src, dst, at = [], [], 0
    for _ in range(128):
        src.append(np.full(300, at)); dst.append(at + 1 + np.arange(300)); at += 301
    for _ in range(6):
        kids = at + 1 + np.arange(50)
        src += [np.full(50, at), np.repeat(kids, 50)]
        dst += [kids, at + 51 + np.arange(2500)]
        at += 2551
    mids = at
    for _ in range(100):
        e = _matchings(rng, 1200, 40) + at
        src.append(e[:, 0]); dst.append(e[:, 1]); at += 1200
    g = gen.csr_from_arcs(at, np.concatenate(src), np.concatenate(dst), directed=False, name="parts")
    deg = g.degrees()
    assert deg[mids:].max() <= 40 and deg[:mids].max() == 300
    ei, ef, er, _ = orc.bcm(g, 1)
    with B.BcmGraph.from_graph(g) as h:
        ids, far, reach, st = h.topk(1, heavy_words=1)
    assert np.array_equal(ids, ei) and np.array_equal(far, ef) and np.array_equal(reach, er)
    assert st["completed"] + st["cut"] == g.n
    stars, trees, leaves = 128 * 600, 6 * 51 * 5100, 6 * 2500
    assert int(deg[mids:].sum()) > 2 * (stars + trees + leaves)
    # (up to a wave of the parts may be searched beside the last tree sources, to level 1 at least)
    assert st["m_vis"] <= stars + trees + leaves + 256 * 40, st
