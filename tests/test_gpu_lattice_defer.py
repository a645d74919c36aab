"""Frontiers longer than the one-source kernel's queues (2^18 entries) on padded
rows: every source of a shard is handed to the grid-wide pass, for rows of 4
and of 8 entries, with and without landmark bounds and at two block shapes,
against the oracle's searches from the same sources.  Whole numbers: exact.
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


@pytest.mark.parametrize("degree", [4, 8])
def test_wide_frontiers_defer(B, gen, orc, degree):
    rng = np.random.default_rng(degree)
    n, shards, k = 1 << 20, 4096, 10
    e = np.concatenate([rng.permutation(n).reshape(-1, 2) for _ in range(degree)])
    g = gen.csr_from_arcs(n, e[:, 0], e[:, 1], directed=False, name="matchings")
    assert g.degrees().max() <= degree
    src = orc.order(g)[B.shard_positions(n, 5, shards)]
    assert 100 < len(src) < 500
    f, r = orc.farness_all(g, sources=src)
    assert (r == n).all()   # so the ranking is by farness, then id
    key = sorted(range(len(src)), key=lambda i: (int(f[i]), int(src[i])))[:k]
    with B.BcmGraph.from_graph(g) as h:
        for kw in (dict(), dict(threads=256), dict(flags=B.BCM_NO_PREFILTER)):
            for _ in range(2):
                ids, far, reach, st = h.topk(k, shard_index=5, shard_count=shards, **kw)
                assert np.array_equal(ids, src[key]) and np.array_equal(far, f[key]) and (reach == n).all(), kw
                assert st["deferred"] > 0, (kw, st)
