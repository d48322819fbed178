"""GPU: runs that go through dedup and stability in several batches.

Dedup takes 4,194,304 units at a time (or one scale), stability as many scales as
1 GiB of scratch holds, the last of them again with the next ones; where the
device has less memory free, two scales at a time.  The results are those of a run
of each scale alone, and of the two covers alone.  The graphs are a 1,000-node
planted partition among isolated nodes, which make the batches large."""
import numpy as np
import pytest

from paper_1301_0955_gb300 import synth
from test_gpu_scale_batches import mscd_mod  # noqa: F401

pytestmark = pytest.mark.gpu


def planted_among(n):
    """Nodes i * (n // 1000) are those of the planted partition."""
    g = synth.config_graph(0)
    step = n // g.n
    rp = np.zeros(n + 1, np.int64)
    rp[np.arange(g.n) * step + 1] = np.diff(g.row_ptr)
    return np.cumsum(rp), (g.col.astype(np.int64) * step).astype(np.int32), step


def test_stability_in_several_chunks(mscd_mod):
    """4,000,003 nodes: 96 MB a scale, 11 scales a chunk."""
    import torch

    mscd = mscd_mod
    n = 4_000_003
    rp, col, step = planted_among(n)
    alphas = np.linspace(0.4, 1.4, 25)
    seeds = (np.arange(0, 1000, 17) * step).astype(np.int32)
    ctx = mscd.Context(0)
    gid = ctx.load_csr(n, rp, col)
    launches = []

    def run():
        at = mscd.load().mscd_launch_count()
        assert ctx.run(gid, alphas, seeds) == mscd.OK
        launches.append(mscd.load().mscd_launch_count() - at)
        return [ctx.communities(s) for s in range(len(alphas))], np.array(ctx.stability()[0])

    covers, nmi = run()
    want = np.array([ctx.nmi_covers(n, covers[s][:2], covers[s + 1][:2]) for s in range(len(alphas) - 1)])
    assert np.array_equal(nmi, want)
    assert len(set(want)) > 5  # the scales differ, on both sides of the seams
    # room for two scales (and the table of terms), not for eleven
    torch.cuda.synchronize()
    hold, left = [], 500 << 20
    try:
        while (free := torch.cuda.mem_get_info()[0]) > left + (64 << 20):
            hold.append(torch.empty(min(free - left, 16 << 30), dtype=torch.uint8, device="cuda"))
        again, nmi2 = run()
    finally:
        hold.clear()
        torch.cuda.empty_cache()
    assert np.array_equal(nmi2, want)
    for a, b in zip(covers, again):
        assert all(np.array_equal(x, y) for x, y in zip(a, b))
    assert launches[1] > launches[0] + 100  # 24 chunks instead of 3
    ctx.free_graph(gid)
    ctx.close()


def test_dedup_in_several_batches(mscd_mod):
    """300,001 seeds: 13 scales a batch."""
    mscd = mscd_mod
    n = 300_001
    rp, col, step = planted_among(n)
    alphas = np.linspace(0.4, 1.4, 16)
    ctx = mscd.Context(0)
    gid = ctx.load_csr(n, rp, col)
    assert ctx.run(gid, alphas) == mscd.OK
    got = [ctx.communities(s) for s in range(len(alphas))]
    nmi = np.array(ctx.stability()[0])
    for s in (0, 12):
        assert nmi[s] == ctx.nmi_covers(n, got[s][:2], got[s + 1][:2])
    for s in (0, 6, 12, 13, 15):
        assert ctx.run(gid, alphas[s:s + 1]) == mscd.OK
        for a, b in zip(got[s], ctx.communities(0)):
            assert np.array_equal(a, b), s
    ctx.free_graph(gid)
    ctx.close()
