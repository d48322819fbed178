"""GPU: initial members added in bulk agree with the oracle, which adds them one
by one: lists around the warp's width, repeats within and across its chunks,
the seed itself, members that fill the slots, in both slot classes."""
import numpy as np
import pytest

from paper_1301_0955_gb300 import synth
from test_gpu_parity import F_RTOL, ctx  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("weighted", [False, True])
@pytest.mark.parametrize("slots", [0, 128])
def test_bulk_initial_members(orc, ctx, weighted, slots):
    from paper_1301_0955_gb300 import mscd

    g = synth.hierarchical_lfr(1200, 12, 60, 2.5, 1.5, (20, 200), (0.3, 0.1), weights=(0.5, 2.0) if weighted else None,
                               seed=77)
    rng = np.random.default_rng(6)
    seeds, lists = [], []
    for m in (0, 1, 2, 31, 32, 33, 64, 100, 700):
        for kind in range(3):
            s = int(rng.integers(g.n))
            x = rng.choice(g.n, m, replace=False)
            if kind == 1:  # every node twice, neighbouring and far apart
                x = np.concatenate([np.repeat(x, 2), x[::-1]])
            if kind == 2:
                x = np.concatenate([[s], x, [s]])
            seeds.append(s)
            lists.append(x)
    seeds = np.array(seeds, np.int32)
    ptr = np.concatenate([[0], np.cumsum([len(x) for x in lists])]).astype(np.int64)
    nodes = np.concatenate(lists).astype(np.int32)
    alphas = np.array([1.0, 0.7])
    G = orc.Graph(g.n, g.row_ptr, g.col, g.w)
    rc, optr, onodes, of, ost = orc.run(G, alphas, seeds, threads=8, init=(ptr, nodes))
    assert rc == 0
    c = mscd.Context(0, smem_slots=slots)
    gid = c.load_csr(g.n, g.row_ptr, g.col, g.w)
    assert c.run_init(gid, alphas, seeds, ptr, nodes) == 0
    N = len(seeds)
    for s in range(len(alphas)):
        p, got, f, st = c.memberships(s)
        sl = slice(s * N, (s + 1) * N)
        assert np.array_equal(p, optr[s * N:(s + 1) * N + 1] - optr[s * N])
        assert np.array_equal(got, onodes[optr[s * N]:optr[(s + 1) * N]])
        np.testing.assert_allclose(f, of[sl], rtol=F_RTOL, atol=0)
        assert np.array_equal(st[:, :6], ost[sl, :6])
    c.close()
