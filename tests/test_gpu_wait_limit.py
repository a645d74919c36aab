"""A wait limit of the default's length or longer changes nothing: the same
kernels run (the same waves and launches) as without one, and exactly; a
shorter one is exact too.
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


def test_the_default_limit_given(B, gen, orc):
    for g in (gen.ba(2000, 3, seed=1), gen.rmat(12, 8, seed=2)):
        f, r = orc.farness_all(g)
        ids = orc.topk(f, r, 10)
        with B.BcmGraph.from_graph(g) as h:
            h.farness_all()
            h.topk(10)
            every, top = h.farness_all(), h.topk(10)
            for limit in (20 * 10 ** 9, 10 ** 12, 10 ** 9):
                a, t = h.farness_all(wait_limit_ns=limit), h.topk(10, wait_limit_ns=limit)
                assert np.array_equal(a[0], f) and np.array_equal(a[1], r)
                assert np.array_equal(t[0], ids) and np.array_equal(t[1], f[ids]) and np.array_equal(t[2], r[ids])
                if limit >= 20 * 10 ** 9:
                    for key in ("waves", "levels", "launches", "m_vis"):
                        assert a[2][key] == every[2][key] and t[3][key] == top[3][key], (limit, key)
