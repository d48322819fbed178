"""GPU: the plain form (one statically mapped unit per warp) where a class's
arena holds fewer units than the call has, and not a multiple of a CTA's four:
every unit is grown once per class."""
import numpy as np
import pytest

from paper_1301_0955_gb300 import synth
from test_gpu_parity import F_RTOL, ctx  # noqa: F401

pytestmark = pytest.mark.gpu


def test_units_beyond_a_chunk(orc, ctx):
    """A weighted hub of 40,000 leaves, 10,000 of them seeds: every unit outgrows
    16,384 slots, of which 4 GiB hold 9,986 (430,080 bytes each).  The scale lets
    a unit join the hub and a few leaves."""
    from paper_1301_0955_gb300 import mscd

    n = 40_001
    rp, col, w = synth.to_csr(n, np.zeros(n - 1, np.int64), np.arange(1, n), np.ones(n - 1, np.float32))
    seeds = np.arange(1, 10_001, dtype=np.int32)
    alphas = np.array([3000.0])
    c = mscd.Context(0, schedule=mscd.SCHED_PER_SCALE)
    gid = c.load_csr(n, rp, col, w)
    assert c.run(gid, alphas, seeds) == 0
    st = c.run_stats()
    assert [(l["cap"], l["units"]) for l in st["launches"]] == [(x, 10_000) for x in (1024, 8192, 16384, 65536)]
    assert st["overflow_units"] == 30_000
    ptr, nodes, f, us = c.memberships(0)
    # the persistent form, and the oracle at some of the seeds
    gid2 = ctx.load_csr(n, rp, col, w)
    assert ctx.run(gid2, alphas, seeds) == 0
    for a, b in zip((ptr, nodes, f, us[:, :6]), ctx.memberships(0)):
        assert np.array_equal(a, b if b.ndim == 1 else b[:, :6])
    pick = np.array([0, 1, 1806, 1807, 9983, 9984, 9985, 9986, 9987, 9999])
    rc, optr, onodes, of, ost = orc.run(orc.Graph(n, rp, col, w), alphas, seeds[pick], threads=8)
    assert rc == 0
    for i, j in enumerate(pick):
        assert np.array_equal(nodes[ptr[j]:ptr[j + 1]], onodes[optr[i]:optr[i + 1]]), j
    np.testing.assert_allclose(f[pick], of, rtol=F_RTOL, atol=0)
    assert np.array_equal(us[pick, :6], ost[:, :6])
    ctx.free_graph(gid2)
    c.close()
