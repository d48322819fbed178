"""GPU: which of the wide classes a list of units takes.  65,536 slots where the
list is more than three times as long as an arena of 131,072-slot states holds
(3 * 903 weighted units), 131,072 at once where it is not; what outgrows the first goes on to the second,
and from there to 524,288.  Against the oracle."""
import numpy as np
import pytest

from paper_1301_0955_gb300 import synth
from test_gpu_parity import F_RTOL, ctx  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("leaves,n,n_seeds,caps", [
    (20_000, 70_001, 2710, [1024, 16384, 65536]),
    (20_000, 70_001, 2709, [1024, 16384, 131072]),
    (70_000, 70_001, 2710, [1024, 16384, 65536, 131072]),
    (70_000, 300_001, 200, [1024, 16384, 131072]),
    (140_000, 300_001, 2710, [1024, 16384, 65536, 131072, 524288]),
    (140_000, 300_001, 3, [1024, 8192, 16384, 131072, 524288]),
])
def test_classes_of_a_list(orc, ctx, leaves, n, n_seeds, caps):
    """Weighted star; a unit joins the centre and a few leaves at this scale and
    touches every leaf."""
    rp, col, w = synth.to_csr(n, np.zeros(leaves, np.int64), np.arange(1, leaves + 1), np.ones(leaves, np.float32))
    seeds = np.linspace(1, leaves, n_seeds).astype(np.int32)
    alphas = np.array([3000.0 * leaves / 40_000])
    gid = ctx.load_csr(n, rp, col, w)
    assert ctx.run(gid, alphas, seeds) == 0
    assert [(l["cap"], l["units"]) for l in ctx.run_stats()["launches"]] == [(c, n_seeds) for c in caps]
    ptr, nodes, f, us = ctx.memberships(0)
    pick = np.unique(np.linspace(0, n_seeds - 1, 9).astype(int))
    rc, optr, onodes, of, ost = orc.run(orc.Graph(n, rp, col, w), alphas, seeds[pick], threads=8)
    assert rc == 0
    for i, j in enumerate(pick):
        assert np.array_equal(nodes[ptr[j]:ptr[j + 1]], onodes[optr[i]:optr[i + 1]]), j
    np.testing.assert_allclose(f[pick], of, rtol=F_RTOL, atol=0)
    assert np.array_equal(us[pick, :6], ost[:, :6])
    ctx.free_graph(gid)
