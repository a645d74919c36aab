"""Whether counts beyond two arcs are summed, decided by the sources that the
tests at levels 0 and 1 leave: none, a few, most, and many leaves beside a hub
at the queue's far end, on graphs below and above 65,536 vertices, undirected
and directed, in shards and with sources picked later.  Exact, against the
oracle's Algorithm 1.
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


def _leaves(gen, n, hubs, seed):
    """A Barabasi-Albert graph with `hubs` stars of leaves hung on far vertices."""
    rng = np.random.default_rng(seed)
    base = gen.ba(n, 3, seed=seed)
    src, dst, at = [np.repeat(np.arange(n), base.degrees())], [base.col], n
    for h in rng.integers(n // 2, n, hubs):
        c = n // (4 * hubs)
        src.append(np.full(c, h))
        dst.append(at + np.arange(c))
        at += c
    return gen.csr_from_arcs(at, np.concatenate(src), np.concatenate(dst), directed=False, name="leaves%d" % n)


@pytest.mark.parametrize("k", [1, 10, 100])
def test_probe(B, gen, orc, k):
    graphs = [gen.ba(30000, 8, seed=1), gen.ba(30000, 3, seed=2), _leaves(gen, 24000, 3, 3), gen.ba(80000, 8, seed=4),
              gen.ba(80000, 3, seed=5), _leaves(gen, 60000, 4, 6), gen.rmat(15, 3, seed=7), gen.rmat(17, 2, seed=8)]
    for g in graphs:
        exp = orc.bcm(g, k, refined=g.directed)[:3]
        with B.BcmGraph.from_graph(g) as h:
            for kw in (dict(), dict(), dict(heavy_words=1), dict(grid_lanes=64, heavy_words=1)):
                got = h.topk(k, **kw)
                assert all(np.array_equal(a, b) for a, b in zip(got, exp)), (g.name, k, kw)
                assert got[3]["completed"] + got[3]["cut"] == g.n, (g.name, kw)
            parts = [h.topk(k, shard_index=i, shard_count=3)[:3] for i in range(3)]
        got = B.bcm_topk_merge(*[np.concatenate([p[j] for p in parts]) for j in range(3)], k)
        assert all(np.array_equal(a, b) for a, b in zip(got, exp)), (g.name, k, "shards")
