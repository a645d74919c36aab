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


def _two_parts(gen, a, b, name):
    src = np.concatenate([np.repeat(np.arange(a.n), a.degrees()), a.n + np.repeat(np.arange(b.n), b.degrees())])
    dst = np.concatenate([a.col.astype(np.int64), a.n + b.col.astype(np.int64)])
    return gen.csr_from_arcs(a.n + b.n, src, dst, directed=False, name=name)


@pytest.mark.parametrize("k", [1, 10, 300])
def test_landmark_bounds(B, gen, orc, k):
    """From 8192 vertices on, sources are stopped by landmark bounds before their search: grids in order and
    relabelled (interior first landmark), components without a landmark, distances that concentrate (the joint
    bound is not taken), rows of 8, and the same without the bounds."""
    graphs = [gen.grid_lcc(100, 95, 0.05, seed=6), gen.relabel(gen.grid_lcc(91, 99, 0.1, seed=7), seed=2),
              _two_parts(gen, gen.grid_lcc(88, 95, 0.02, seed=8), gen.grid_lcc(90, 92, 0.02, seed=9), "two grids"),
              _matchings(gen, 9001, 3, 4), _matchings(gen, 8200, 7, 5), gen.cycle(8192), gen.grid(9000, 1)]
    for g in graphs:
        ei, ef, er, _ = orc.bcm(g, k)
        with B.BcmGraph.from_graph(g) as h:
            for flags in (0, B.BCM_NO_PREFILTER):
                ids, far, reach, st = h.topk(k, flags=flags)
                assert np.array_equal(ids, ei) and np.array_equal(far, ef) and np.array_equal(reach, er), (g.name, flags)
                assert st["sparse"] == g.n and st["completed"] + st["cut"] == g.n, (g.name, st)
            parts = [h.topk(k, shard_index=i, shard_count=2)[:3] for i in range(2)]
        ids, far, reach = B.bcm_topk_merge(*[np.concatenate([q[j] for q in parts]) for j in range(3)], k)
        assert np.array_equal(ids, ei) and np.array_equal(far, ef) and np.array_equal(reach, er), (g.name, "shards")


def test_landmark_distances_too_large(B, gen):
    """A path longer than the bounds' distance limit (65,535): the middle vertices, from the closed form."""
    n = 70001
    with B.BcmGraph.from_graph(gen.path(n)) as h:
        ids, far, reach, _ = h.topk(3)
    m = n // 2
    assert ids.tolist() == [m, m - 1, m + 1] and (reach == n).all()
    assert far.tolist() == [m * (m + 1), m * (m + 1) + 1, m * (m + 1) + 1]


def test_landmark_bounds_in_a_batch(B, gen, orc):
    """Recorded runs (a lattice of this size still fits a batch) give the same answer on every replay."""
    import torch
    graphs = [gen.grid_lcc(96, 92, 0.05, seed=11), gen.grid_lcc(99, 90, 0.1, seed=12)]
    hs = [B.BcmGraph.from_graph(g) for g in graphs]
    out = [[torch.zeros(10, dtype=t, device="cuda") for t in (torch.int32, torch.int64, torch.int32)] for _ in graphs]
    batch = B.BcmBatch([h.h for h in hs], [10, 10], out, torch.cuda.Stream())
    for _ in range(2):
        for o in out:
            for t in o:
                t.zero_()
        torch.cuda.synchronize()
        batch.run()
        for g, o in zip(graphs, out):
            ei, ef, er, _ = orc.bcm(g, 10)
            assert np.array_equal(o[0].cpu().numpy(), ei) and np.array_equal(o[1].cpu().numpy(), ef)
            assert np.array_equal(o[2].cpu().numpy(), er)
    batch.close()
