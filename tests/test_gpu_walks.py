"""Walk bounds (the prefilter's counts of walks that never turn straight
back) against the oracle: top-k on simple graphs of every size class -- one
seed wave (small graphs, counts kept between runs), grid-wide waves with the
prefilter after the first and sources picked against the threshold by then --
with degrees from 2 (many walk levels matter) to hubs past a warp's and a
block's row limits, digraphs (bounds at both ends of the reach range), shards
and k larger than a wave.  Whole numbers, so every comparison is exact.
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


def _check(got, exp, what):
    for a, b in zip(got, exp):
        assert np.array_equal(a, b), what


@pytest.mark.parametrize("k", [1, 10, 100, 300])
def test_small_graphs(B, gen, orc, k):
    graphs = [gen.ba(1500, 2, seed=100), gen.ba(3000, 8, seed=12), gen.ba(2003, 1, seed=5), gen.rmat(11, 6, seed=3),
              gen.chung_lu(5000, 6.0, 2.3, seed=4), gen.gnp(900, 0.02, seed=8, directed=True), gen.star(2500),
              gen.disjoint_union(gen.ba(700, 2, seed=1), gen.ba(600, 3, seed=2), gen.empty(5))]
    for g in graphs:
        exp = orc.topk_exhaustive(g, k)
        with B.BcmGraph.from_graph(g) as h:
            for kw in ({}, dict(lanes=128), dict(lanes=256, flags=B.BCM_NO_FOOTNOTE), {}):
                ids, far, reach, st = h.topk(k, **kw)
                _check((ids, far, reach), exp, (g.name, k, kw))
                assert st["completed"] + st["cut"] == g.n, (g.name, st)
            h.trim()
            _check(h.topk(k)[:3], exp, (g.name, k, "after trim"))


@pytest.mark.parametrize("k", [1, 100])
def test_grid_wide_graphs(B, gen, orc, k):
    graphs = [gen.ba(20000, 2, seed=7), gen.ba(40000, 4, seed=8), gen.chung_lu(30000, 6.0, 2.3, seed=9),
              gen.rmat(15, 6, seed=10)]
    for g in graphs:
        assert g.degrees().max() > 32
        exp = orc.bcm(g, k, refined=g.directed)[:3]
        with B.BcmGraph.from_graph(g) as h:
            for kw in ({}, dict(grid_lanes=64), dict(grid_lanes=256, flags=B.BCM_NO_FOOTNOTE), dict(heavy_words=1),
                       dict(heavy_words=1 << 30), dict(cta_table=1024), dict(cta_table=1 << 30)):
                ids, far, reach, st = h.topk(k, **kw)
                _check((ids, far, reach), exp, (g.name, k, kw))
            parts = [h.topk(k, shard_index=i, shard_count=2)[:3] for i in range(2)]
        got = B.bcm_topk_merge(*[np.concatenate([p[j] for p in parts]) for j in range(3)], k)
        _check(got, exp, (g.name, k, "shards"))


def test_rows_for_a_whole_block(B, gen, orc):
    """Hubs of more than 1,024 arcs on a graph large enough for the heavy-row list."""
    rng = np.random.default_rng(5)
    n = 20000
    base = gen.ba(n, 2, seed=3)
    src = np.repeat(np.arange(n), base.degrees())
    hub = np.concatenate([np.full(c, v) for v, c in ((0, 9000), (17, 3000), (31, 1500), (19999, 2000))])
    g = gen.csr_from_arcs(n, np.concatenate([src, hub]), np.concatenate([base.col, rng.integers(0, n, hub.size)]),
                          directed=False, name="hubs")
    exp = orc.bcm(g, 10)[:3]
    with B.BcmGraph.from_graph(g) as h:
        _check(h.topk(10)[:3], exp, "hubs")
