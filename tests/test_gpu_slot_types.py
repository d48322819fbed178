"""GPU: the slot layouts and classes at their edges agree with the oracle.

A hub joined to every node decides the layout (d_in and degree in 15 bits each
up to degree 32,767, in 32 bits from 32,768 on) and, once it is in a community,
brings all its neighbours into the slots: 12,000 of them fit the 16,384-slot
class, 32,768 only the wide ones.  Initial communities holding every other node
bring the hub's d_in up to its degree."""
import numpy as np
import pytest

from paper_1301_0955_gb300 import synth
from test_gpu_parity import F_RTOL, ctx  # noqa: F401

pytestmark = pytest.mark.gpu


def hub_graph(h):
    """Node 0 joined to 1..h; the others in cliques of 5."""
    iu, ju = [np.zeros(h, np.int64)], [np.arange(1, h + 1)]
    for d in range(1, 5):
        i = np.arange(1, h + 1 - d)
        i = i[(i - 1) // 5 == (i + d - 1) // 5]
        iu.append(i)
        ju.append(i + d)
    return h + 1, *synth.to_csr(h + 1, np.concatenate(iu), np.concatenate(ju))


@pytest.mark.parametrize("h", [7, 12000, 32767, 32768])
def test_hub_degree_and_classes(orc, ctx, h):
    n, rp, col, _ = hub_graph(h)
    G = orc.Graph(n, rp, col)
    seeds = np.array([0, 1, h, 0, 3], np.int32)
    lists = [[], [], [], list(range(1, h + 1)), list(range(1, h + 1))]
    ptr = np.concatenate([[0], np.cumsum([len(x) for x in lists])]).astype(np.int64)
    nodes = np.concatenate(lists).astype(np.int32)
    alphas = np.array([1.0, 0.6])
    rc, optr, onodes, of, ost = orc.run(G, alphas, seeds, threads=8, init=(ptr, nodes))
    assert rc == 0
    gid = ctx.load_csr(n, rp, col)
    assert ctx.graph_degrees(gid).max() == max(h, 5)
    assert ctx.run_init(gid, alphas, seeds, ptr, nodes) == 0
    N = len(seeds)
    for s in range(len(alphas)):
        p, got, f, st = ctx.memberships(s)
        assert np.array_equal(p, optr[s * N:(s + 1) * N + 1] - optr[s * N])
        assert np.array_equal(got, onodes[optr[s * N]:optr[(s + 1) * N]])
        np.testing.assert_allclose(f, of[s * N:(s + 1) * N], rtol=F_RTOL, atol=0)
        assert np.array_equal(st[:, :6], ost[s * N:(s + 1) * N, :6])
    caps = [l["cap"] for l in ctx.run_stats()["launches"]]
    assert (16384 in caps) == (h >= 12000)
    assert any(c > 16384 for c in caps) == (h > 16384)
    ctx.free_graph(gid)


@pytest.mark.parametrize("h", [60000, 530000])
def test_wide_classes(orc, ctx, h):
    """Group bounds of the wide classes: in shared memory (65,536 slots), in the
    arena (1,048,576 slots: a unit's bounds exceed an SM's shared memory).  The
    initial community holds all nodes but two."""
    n, rp, col, _ = hub_graph(h)
    G = orc.Graph(n, rp, col)
    seeds = np.array([0], np.int32)
    nodes = np.arange(1, h - 1, dtype=np.int32)
    ptr = np.array([0, nodes.size], np.int64)
    alphas = np.array([1.0])
    rc, optr, onodes, of, ost = orc.run(G, alphas, seeds, threads=8, init=(ptr, nodes))
    assert rc == 0
    gid = ctx.load_csr(n, rp, col)
    assert ctx.run_init(gid, alphas, seeds, ptr, nodes) == 0
    p, got, f, st = ctx.memberships(0)
    assert np.array_equal(p, optr) and np.array_equal(got, onodes)
    np.testing.assert_allclose(f, of, rtol=F_RTOL, atol=0)
    assert np.array_equal(st[:, :6], ost[:, :6])
    ctx.free_graph(gid)
