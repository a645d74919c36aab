"""Digraphs whose longest rows are shared by blocks: rows of one part, of parts
with a remainder, of hundreds of parts, more rows than the list holds, and none;
the SCCs, the reach bounds and the top-k against the oracle.  Whole numbers:
exact.
"""
import time

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


def _rows(gen, n, lengths, seed):
    """Vertex i with lengths[i] random out-arcs, the rest with one or two."""
    rng = np.random.default_rng(seed)
    src = [np.repeat(np.arange(n), 2)]
    dst = [rng.integers(0, n, 2 * n)]
    for v, c in enumerate(lengths):
        src.append(np.full(c, v))
        dst.append(rng.permutation(n)[:c])
    return gen.csr_from_arcs(n, np.concatenate(src), np.concatenate(dst), directed=True, name="rows%d" % seed)


@pytest.mark.parametrize("lengths", [[2047, 2049, 4096, 4097, 8192, 40000, 199999], [], [3000] * 70,
                                     [150000] + [2500] * 33])
def test_long_rows(B, gen, orc, lengths):
    g = _rows(gen, 200000, lengths, len(lengths))
    comp, al, om, nc = orc.alpha_omega_refined(g)
    with B.BcmGraph.from_graph(g) as h:
        lab, lo, hi, count = h.scc_bounds()
    assert count == nc and np.array_equal(lo, al) and np.array_equal(hi, om)
    pairs = np.unique(np.stack([lab.astype(np.int64), np.asarray(comp).astype(np.int64)], 1), axis=0)
    assert len(pairs) == nc


def test_more_rows_than_the_list_holds(B, gen, orc):
    """4,200 rows of 2,100 arcs: the last hundred stay with their warps."""
    n, rows = 6000, 4200
    src = np.repeat(np.arange(rows), 2100)
    dst = (src * 7 + np.tile(np.arange(2100), rows) * 2 + 1) % n
    g = gen.csr_from_arcs(n, src, dst, directed=True, name="many")
    assert (np.sort(g.degrees())[-4150:] > 2048).all()
    comp, al, om, nc = orc.alpha_omega_refined(g)
    with B.BcmGraph.from_graph(g) as h:
        lab, lo, hi, count = h.scc_bounds()
    assert count == nc and np.array_equal(lo, al) and np.array_equal(hi, om)


def _scc_time(B, gen, n, src, dst):
    """The best of 20 whole calls (handle, SCCs and bounds, release), and alpha."""
    import torch
    g = gen.csr_from_arcs(n, src, dst, directed=True, name="rows")
    rp = torch.from_numpy(g.row_ptr.view(np.int64)).cuda()
    col = torch.from_numpy(g.col.view(np.int32)).cuda()
    out = [torch.zeros(n, dtype=torch.int32, device="cuda") for _ in range(3)]
    best = np.inf
    for _ in range(20):
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        with B.BcmGraph(rp, col, n, True, on_device=True) as h:
            assert B.bcm_scc_bounds(h.h, *out, out_on_device=True) == n
        best = min(best, (time.perf_counter() - t0) * 1e3)
    return best, out[1].cpu().numpy()


def test_one_row_of_a_million(B, gen):
    """Its time against that of the same arcs in rows of 2,000, which are short: the whole grid on the row took as long,
    four blocks on it half as long again, so a quarter more is the bound."""
    n, m = 1200000, 1000000
    one, lo = _scc_time(B, gen, n, np.zeros(m, np.int64), np.arange(1, m + 1))
    assert lo[0] == m + 1 and (lo[1:] == 1).all()   # (the first of the largest SCCs: its reach is measured)
    many, _ = _scc_time(B, gen, n, np.repeat(np.arange(500), 2000), np.arange(500, m + 500))
    assert one < 1.25 * many, (one, many)
