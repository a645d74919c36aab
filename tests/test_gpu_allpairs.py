"""All pairs (lanes are targets, a cluster per wave) against the oracle:
every vertex's farness and reach, and the top-k of small graphs from them, at
sizes around a lane word, a CTA's and a cluster's waves, with every lane
width; rows for a thread, a warp and a CTA; digraphs, unreachable parts,
self-loops and repeats, tied ranks; and the entry point without allocation,
with its rows laid out by degree and as given.  Whole numbers: exact.
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


def _graphs(gen):
    return [gen.path(2), gen.path(63), gen.cycle(64), gen.star(65), gen.gnp(127, 0.03, seed=1, directed=True),
            gen.gnp(257, 0.02, seed=2, directed=False), gen.complete(129), gen.dpath(200), gen.star(6000),
            gen.with_self_loops_and_repeats(gen.ba(1000, 3, seed=3), seed=4), gen.rmat(12, 8, seed=5),
            gen.disjoint_union(gen.ba(900, 2, seed=6), gen.cycle(64), gen.empty(3), gen.ba(500, 4, seed=7)),
            gen.chung_lu(9729, 6.0, 2.3, seed=8), gen.rmat(14, 4, seed=9)]


def _noalloc(B, g):
    import torch
    rp = torch.from_numpy(g.row_ptr.astype(np.int64)).cuda()
    col = torch.from_numpy(g.col.astype(np.int32)).cuda()
    far = torch.full((g.n,), -1, dtype=torch.int64, device="cuda")
    reach = torch.full((g.n,), -1, dtype=torch.int32, device="cuda")
    B.bcm_farness_all_noalloc(rp, col, g.n, g.m, None, far, reach)
    return far.cpu().numpy().astype(np.uint64), reach.cpu().numpy().astype(np.uint32)


@pytest.mark.parametrize("lanes", [0, 64, 128, 256])
def test_every_vertex(B, gen, orc, lanes):
    for g in _graphs(gen):
        f, r = orc.farness_all(g)
        with B.BcmGraph.from_graph(g) as h:
            for _ in range(2):
                gf, gr, st = h.farness_all(grid_lanes=lanes)
                assert np.array_equal(gf, f) and np.array_equal(gr, r), (g.name, lanes)
                assert st["completed"] == g.n
            h.trim()
            gf, gr, _ = h.farness_all(grid_lanes=lanes)
            assert np.array_equal(gf, f) and np.array_equal(gr, r), (g.name, lanes, "after trim")
        if lanes == 0:
            gf, gr = _noalloc(B, g)
            assert np.array_equal(gf, f) and np.array_equal(gr, r), (g.name, "without allocation")


@pytest.mark.parametrize("k", [1, 33, 1024])
def test_topk_from_every_vertex(B, gen, orc, k):
    for g in _graphs(gen):
        exp = orc.topk_exhaustive(g, k)
        with B.BcmGraph.from_graph(g) as h:
            for _ in range(2):
                ids, far, reach, st = h.topk(k)
                assert np.array_equal(ids, exp[0]) and np.array_equal(far, exp[1]) and np.array_equal(reach, exp[2]), \
                    (g.name, k)
            # the kernels that search from sources give the same
            ids, far, reach, st = h.topk(k, lanes=128)
            assert np.array_equal(ids, exp[0]) and np.array_equal(far, exp[1]), (g.name, k)
