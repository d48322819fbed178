"""GPU: the growth's choices by size agree with the oracle: left-over units in
shared memory (at most one an SM) or in the arenas, and ranking ties settled by
whole numbers (alpha = 1, and 1/2 below 2^31) or by the logarithms."""
import numpy as np
import pytest

from paper_1301_0955_gb300 import synth
from test_gpu_parity import compare_units, ctx, oracle_graph  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("weighted", [False, True])
@pytest.mark.parametrize("n_seeds", [1, 31, 400])
def test_left_over_units(orc, ctx, n_seeds, weighted):
    """64-slot first class: almost every unit goes on to the 512- and 4,096-slot
    classes, a few of them in shared memory, many in the arenas."""
    from paper_1301_0955_gb300 import mscd

    c = mscd.Context(0, smem_slots=64)
    g = synth.hierarchical_lfr(3000, 18, 90, 2.5, 1.5, (20, 300), (0.3, 0.1),
                               weights=(0.5, 2.0) if weighted else None, seed=31)
    G = oracle_graph(orc, g)
    seeds = np.linspace(0, g.n - 1, n_seeds).astype(np.int32)
    alphas = np.array([0.5])
    gid = c.load_csr(g.n, g.row_ptr, g.col, g.w)
    assert c.run(gid, alphas, seeds) == 0
    wide = [l for l in c.run_stats()["launches"] if l["cap"] == 4096]
    assert wide and wide[0]["smem"] == (1 if wide[0]["units"] <= 152 else 0)
    compare_units(orc, c, G, alphas, seeds, threads=8)
    c.close()


@pytest.mark.parametrize("scale", [1.0, 2.0 ** 20])
def test_ranking_ties(orc, ctx, scale):
    """Weights from {1, 2, 4} times `scale`, one edge of weight 1 keeping the unit
    at 1: d_in and degrees below and above 2^31, ties at every step."""
    rng = np.random.default_rng(9)
    n = 240
    iu, ju = np.triu_indices(n, 1)
    keep = (rng.random(iu.size) < 0.1) | (ju == iu + 1)
    w = (rng.choice([1.0, 2.0, 4.0], int(keep.sum())) * scale * (1024.0 if scale > 1 else 1.0)).astype(np.float32)
    w[0] = 1.0
    rp, col, ww = synth.to_csr(n, iu[keep], ju[keep], w)
    G = orc.Graph(n, rp, col, ww)
    gid = ctx.load_csr(n, rp, col, ww)
    assert (ctx.graph_degrees(gid).max() >= 2 ** 31) == (scale > 1)
    alphas = np.array([1.0, 0.5, 0.75])
    seeds = np.arange(0, n, 5, dtype=np.int32)
    assert ctx.run(gid, alphas, seeds) == 0
    compare_units(orc, ctx, G, alphas, seeds, threads=8)
    ctx.free_graph(gid)
