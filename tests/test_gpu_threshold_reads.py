"""bcm_topk_threshold while a small graph's run publishes its k-th key from
every vertex's farness: each snapshot is no key or the final one, never a
mixture.  Whole numbers: exact.
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


def test_reads_while_publishing(B, gen, orc):
    import torch
    g, k = gen.ba(2000, 3, seed=1), 10
    ids, far, reach = orc.topk_exhaustive(g, k)
    final = (1, (int(reach[-1]) - 1) ** 2, int(far[-1]), int(ids[-1]))
    out = [np.zeros(k, t) for t in (np.uint32, np.uint64, np.uint32)]
    reads = 0
    with B.BcmGraph.from_graph(g, stream=torch.cuda.Stream().cuda_stream) as h:
        for _ in range(300):
            B.bcm_topk_start(h.h, k, None, *out)
            while not B.bcm_topk_finish(h.h, wait=False):
                t = B.bcm_topk_threshold(h.h)
                assert not t[0] or t == final
                reads += 1
            assert B.bcm_topk_threshold(h.h) == final
            assert np.array_equal(out[0], ids) and np.array_equal(out[1], far) and np.array_equal(out[2], reach)
    assert reads > 0
