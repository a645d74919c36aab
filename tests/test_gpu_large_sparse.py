"""Graphs too large for any shape of the all-pairs kernel, by default and with
256 lanes: the workspace is told and every vertex's farness is exact.
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


@pytest.mark.parametrize("n,lanes", [(5000000, 0), (1400000, 256)])
def test_no_shape_fits(B, gen, n, lanes):
    a = np.arange(0, 3000, 3)   # 1,000 paths of three vertices, the rest alone
    g = gen.csr_from_arcs(n, np.concatenate([a, a + 1]), np.concatenate([a + 1, a + 2]), directed=True, name="paths")
    f, r = np.zeros(n, np.uint64), np.ones(n, np.uint32)
    f[a], f[a + 1], r[a], r[a + 1] = 3, 1, 3, 2
    with B.BcmGraph.from_graph(g) as h:
        assert B.bcm_workspace_bytes(h.h, B.make_options(grid_lanes=lanes)) > 0
        gf, gr, st = h.farness_all(grid_lanes=lanes)
    assert np.array_equal(gf, f) and np.array_equal(gr, r) and st["completed"] == n
