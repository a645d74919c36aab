"""A batch and runs of its graphs by themselves, in turn: a replay must not see
what a run with other options left in a workspace (other kernels, other
layouts, larger slots), nor the run what the replay left, and a replay's
workspace must not have passed on to another graph.  Graphs whose recorded
runs are all pairs, per-CTA waves (too dense for all pairs) and the one-source
kernel; used before and after the batch is made, trimmed between replays.
Whole numbers, so every comparison is exact.
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


@pytest.mark.parametrize("before", [False, True])
def test_runs_between_replays(B, gen, orc, before):
    import torch
    graphs = [gen.ba(2000, 3, seed=1), gen.ba(9000, 30, seed=2), gen.grid_lcc(96, 92, 0.05, seed=11),
              gen.rmat(12, 8, seed=5)]
    assert graphs[1].n * graphs[1].m // 64 > 1 << 26
    other = gen.chung_lu(9000, 6.0, 2.3, seed=4)
    k = 10
    exp, every = [], []
    for g in graphs + [other]:
        f, r = orc.farness_all(g)
        ids = orc.topk(f, r, k)
        every.append((f, r))
        exp.append((ids, f[ids], r[ids]))
    hs = [B.BcmGraph.from_graph(g) for g in graphs]
    third = B.BcmGraph.from_graph(other)
    runs = [dict(flags=B.BCM_TRACE), dict(flags=B.BCM_NO_PREFILTER), dict(lanes=128), dict(flags=B.BCM_NO_DEFER),
            dict(wait_limit_ns=10 ** 9), dict(flags=B.BCM_SPARSE), dict()]

    def direct(h, i, kw):
        got = h.topk(k, **kw)[:3]
        assert all(np.array_equal(a, b) for a, b in zip(got, exp[i])), (i, kw)

    def replay(what):
        for o in outs:
            for t in o:
                t.fill_(-1)
        torch.cuda.synchronize()
        batch.run()
        for o, e, g in zip(outs, exp, graphs):
            assert np.array_equal(o[0].cpu().numpy().view(np.uint32), e[0]), (what, g.name)
            assert np.array_equal(o[1].cpu().numpy().view(np.uint64), e[1]), (what, g.name)
            assert np.array_equal(o[2].cpu().numpy().view(np.uint32), e[2]), (what, g.name)

    if before:
        for i, h in enumerate(hs):
            direct(h, i, runs[0])
    outs = [tuple(torch.zeros(k, dtype=t, device="cuda") for t in (torch.int32, torch.int64, torch.int32))
            for _ in graphs]
    batch = B.BcmBatch([h.h for h in hs], [k] * len(hs), outs, torch.cuda.Stream())
    replay("first")
    for kw in runs:
        for i, h in enumerate(hs):
            direct(h, i, kw)
            direct(third, len(hs), kw)
        replay(kw)
        for i, h in enumerate(hs):
            direct(h, i, runs[0])
    for i, h in enumerate(hs):
        gf, gr, _ = h.farness_all()
        assert np.array_equal(gf, every[i][0]) and np.array_equal(gr, every[i][1]), graphs[i].name
    replay("every vertex")
    for h in hs:
        h.trim()
    for _ in range(2):
        direct(third, len(hs), runs[0])
        third.trim()
    replay("trimmed")
    for i, h in enumerate(hs):
        direct(h, i, runs[1])
        direct(h, i, {})
    batch.close()
    for i, h in enumerate(hs):
        direct(h, i, {})
        h.trim()
        direct(h, i, runs[0])
        h.close()
    third.close()
