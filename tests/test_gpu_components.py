"""Components (r(v) and labels) where they are found from the largest-degree
vertex's marks, against the oracle: a hub whose component is the graph, most of
it, less than half of it (the marks are dropped) or far from it (a long tail),
many small components beside it, isolated vertices, and hubs just below and at
the degree from which marks are tried.  Whole numbers: exact.
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
    u = gen.disjoint_union
    tail = gen.csr_from_arcs(3000, np.r_[np.zeros(100, np.int64), np.arange(100, 2999)],
                             np.r_[np.arange(1, 101), np.arange(101, 3000)], directed=False, name="broom")
    return [gen.star(64), gen.star(65), gen.star(66), gen.chung_lu(20000, 4.0, 2.3, seed=1), gen.ba(5000, 2, seed=2),
            u(gen.star(200), gen.grid(60, 60)), u(gen.grid(40, 40), gen.star(1700), gen.empty(50)), tail,
            gen.relabel(u(gen.chung_lu(4000, 3.0, 2.3, seed=3), gen.cycle(900), gen.star(120)), seed=4),
            u(gen.empty(500), gen.star(100), gen.star(100)),
            gen.with_self_loops_and_repeats(gen.chung_lu(3000, 5.0, 2.3, seed=5), seed=6)]


def test_components(B, gen, orc):
    for g in _graphs(gen):
        comp, n_comp = orc.scc(g)
        comp = np.asarray(comp)
        size = np.bincount(comp)[comp]
        with B.BcmGraph.from_graph(g) as h:
            order, lo, hi = h.preprocess()
            lab, al, om, nc = h.scc_bounds()
        assert np.array_equal(order, orc.order(g)), g.name
        assert np.array_equal(lo, size) and np.array_equal(hi, size) and nc == n_comp, g.name
        # the same partition, labels in order of the smallest member
        first = np.full(nc, g.n)
        np.minimum.at(first, lab, np.arange(g.n))
        assert (np.diff(first) > 0).all() and len(set(zip(lab.tolist(), comp.tolist()))) == nc, g.name
