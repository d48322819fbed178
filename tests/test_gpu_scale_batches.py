"""GPU: all the scales of a run deduplicated, and compared, in the same launches.

A batch of scales keeps its communities side by side in one block and takes
all pairs of scales through each launch.  Each scale must come out as from a
run of that scale alone, and each pair's stability as from the two covers
alone: the same terms rounded once and added as integers, so the same bits.
"""
import numpy as np
import pytest

from paper_1301_0955_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mscd_mod():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1301_0955_gb300 import build, mscd

    build.build()
    return mscd


@pytest.mark.parametrize("bits", [0, 2])
@pytest.mark.parametrize("n_scales,seeds", [(1, [3]), (2, [0]), (3, [7, 7, 500]), (33, list(range(0, 1000, 31))),
                                            (70, list(range(129)))])
def test_batched_scales_equal_single_scales(mscd_mod, n_scales, seeds, bits):
    mscd = mscd_mod
    g = synth.config_graph(0)
    alphas = np.linspace(0.5, 1.3, n_scales)
    seeds = np.array(seeds, np.int32)
    ctx = mscd.Context(0, list_hash_bits=bits)
    gid = ctx.load_csr(g.n, g.row_ptr, g.col)
    assert ctx.run(gid, alphas, seeds) == mscd.OK
    got = [ctx.communities(s) for s in range(n_scales)]
    nmi = ctx.stability()[0]
    assert len(nmi) == n_scales - 1
    for s in range(n_scales):
        assert ctx.run(gid, alphas[s : s + 1], seeds) == mscd.OK
        for a, b in zip(got[s], ctx.communities(0)):
            assert np.array_equal(a, b), s
    want = [ctx.nmi_covers(g.n, got[s][:2], got[s + 1][:2]) for s in range(n_scales - 1)]
    assert np.array_equal(np.array(nmi), np.array(want), equal_nan=True)
    ctx.free_graph(gid)
    ctx.close()
