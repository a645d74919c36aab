"""bcm_graph_trim gives back what a run laid out for itself: other graphs of the
same size then run without new device memory.  The rows by degree (all
pairs), the padded rows of a lattice and the walk counts are each far larger
than the margin.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

MARGIN = 8 << 20


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


def _dense(gen, seed):
    rng = np.random.default_rng(seed)
    n, m = 40000, 6000000
    return gen.csr_from_arcs(n, rng.integers(0, n, m), rng.integers(0, n, m), directed=False, name="dense")


@pytest.mark.parametrize("what", ["rows", "lattice"])
def test_trim_gives_back(B, gen, what):
    import torch
    if what == "rows":
        g = _dense(gen, 1)
        run = lambda h: h.farness_all()
        assert 4 * g.m > 4 * MARGIN
    else:
        g = gen.grid_lcc(1024, 1024, 0.05, seed=1)
        run = lambda h: h.topk(1)
        assert 16 * g.n + MARGIN // 2 > 2 * MARGIN
    hs = [B.BcmGraph.from_graph(g) for _ in range(6)]
    for h in hs:
        h.preprocess()
    first = run(hs[0])
    hs[0].trim()
    before = torch.cuda.mem_get_info()[0]
    for h in hs[1:] + hs[:1]:      # (six: preprocessing's scratch is in the pool too, and serves the first few)
        got = run(h)
        h.trim()
        assert all(np.array_equal(x, y) for x, y in zip(first[:-1], got[:-1]))
    after = torch.cuda.mem_get_info()[0]
    assert before - after < MARGIN, (before, after)
    for h in hs:
        h.close()
