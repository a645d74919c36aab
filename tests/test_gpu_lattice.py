"""The one-source kernel on padded rows (undirected graphs of largest degree
at most 8) against the oracle, where it can go wrong: rows of 4 and of 8
entries, frontiers longer than the queue part in shared memory, the bitmap in
global memory, self-loops and repeated arcs, every block shape, all vertices
(no cut) and shards.  Whole numbers, so every comparison is exact.
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


def _matchings(gen, n, d, seed):
    """d random perfect matchings: degrees at most d, frontiers of about half the graph."""
    rng = np.random.default_rng(seed)
    p = [rng.permutation(n - n % 2).reshape(-1, 2) for _ in range(d)]
    e = np.concatenate(p)
    return gen.csr_from_arcs(n, e[:, 0], e[:, 1], directed=False, name="matchings_n%d_d%d" % (n, d))


def _graphs(gen):
    return [_matchings(gen, 6001, 3, 1), _matchings(gen, 6000, 4, 2), _matchings(gen, 5003, 8, 3),
            gen.grid_lcc(70, 61, 0.1, seed=2), gen.cycle(4097), gen.path(4100),
            gen.with_self_loops_and_repeats(gen.grid(65, 67), seed=3, frac=0.02)]


@pytest.mark.parametrize("threads", [0, 128, 256, 512, 1024])
def test_padded_rows_topk(B, gen, orc, threads):
    for g in _graphs(gen):
        assert g.degrees().max() <= 8
        with B.BcmGraph.from_graph(g) as h:
            for k in (1, 10, 300):
                ei, ef, er, _ = orc.bcm(g, k)
                ids, far, reach, st = h.topk(k, threads=threads)
                assert np.array_equal(ids, ei) and np.array_equal(far, ef) and np.array_equal(reach, er), (g.name, k)
                assert st["sparse"] == g.n and st["completed"] + st["cut"] == g.n, (g.name, st)


def test_padded_rows_every_vertex(B, gen, orc):
    for g in _graphs(gen)[:4]:
        f, r = orc.farness_all(g)
        with B.BcmGraph.from_graph(g) as h:
            gf, gr, _ = h.farness_all(flags=B.BCM_SPARSE)
        assert np.array_equal(gf, f) and np.array_equal(gr, r), g.name


def test_padded_rows_shards(B, gen, orc):
    g = gen.grid_lcc(90, 75, 0.05, seed=8)
    ei, ef, er, _ = orc.bcm(g, 20)
    with B.BcmGraph.from_graph(g) as h:
        parts = [h.topk(20, shard_index=i, shard_count=3)[:3] for i in range(3)]
    ids, far, reach = B.bcm_topk_merge(*[np.concatenate([p[j] for p in parts]) for j in range(3)], 20)
    assert np.array_equal(ids, ei) and np.array_equal(far, ef) and np.array_equal(reach, er)


def test_bitmap_in_global_memory(B, gen, orc):
    """More vertices than the shared-memory bitmap holds: 220,000 cycles of 8 and a damaged grid."""
    g = gen.grid_lcc(40, 43, 0.1, seed=5)
    c = 220000
    v = np.arange(8 * c, dtype=np.int64)
    nxt = (v // 8) * 8 + (v + 1) % 8
    src = np.concatenate([np.repeat(np.arange(g.n), g.degrees()), v + g.n])
    dst = np.concatenate([g.col.astype(np.int64), nxt + g.n])
    big = gen.csr_from_arcs(g.n + 8 * c, src, dst, directed=False, name="grid_and_cycles")
    ei, ef, er, _ = orc.bcm(big, 10)
    with B.BcmGraph.from_graph(big) as h:
        ids, far, reach, st = h.topk(10)
    assert np.array_equal(ids, ei) and np.array_equal(far, ef) and np.array_equal(reach, er)
    assert st["sparse"] == big.n
