"""GPU: symmetry found by counting.  A load looks up the partners of the entries
above the diagonal only; entries below it without a partner are found by their
number.  Statuses against the oracle's, device and host arrays."""
import numpy as np
import pytest

from paper_1301_0955_gb300 import synth
from test_gpu_parity import ctx  # noqa: F401

pytestmark = pytest.mark.gpu


def drop(rp, col, w, e):
    """The CSR without entry e."""
    row = int(np.searchsorted(rp, e, side="right")) - 1
    r = rp.copy()
    r[row + 1:] -= 1
    return r, np.delete(col, e), None if w is None else np.delete(w, e)


@pytest.mark.parametrize("weighted", [False, True])
@pytest.mark.parametrize("kind", ["whole", "no upper entry", "no lower entry", "both", "lower weight", "upper weight",
                                  "range"])
def test_symmetry(orc, ctx, kind, weighted):
    import torch

    if not weighted and ("weight" in kind or kind == "range"):
        pytest.skip("weights only")
    g = synth.hierarchical_lfr(700, 30, 300, 2.5, 1.5, (20, 200), (0.3, 0.1), weights=(0.5, 2.0) if weighted else None,
                               seed=5)
    rp, col, w = g.row_ptr.copy(), g.col.copy(), None if g.w is None else g.w.copy()
    row = np.repeat(np.arange(g.n), np.diff(rp))
    up, low = np.flatnonzero(col > row), np.flatnonzero(col < row)
    if kind in ("no upper entry", "both"):
        rp, col, w = drop(rp, col, w, int(up[len(up) // 2]))
    if kind in ("no lower entry", "both"):  # of another pair: as many above as below are left
        rp, col, w = drop(rp, col, w, int(low[len(low) // 3]))
    if kind == "lower weight":
        w[low[7]] *= 2
    if kind == "upper weight":
        w[up[7]] *= 2
    if kind == "range":  # totals beyond 62 bits, every entry fine by itself
        w[:] = 2.0 ** 40
        w[0] = w[low[np.flatnonzero((row[low] == col[0]) & (col[low] == 0))[0]]] = 2.0 ** -20
    want = orc.Graph(g.n, rp, col, w).status
    got, gid = ctx.try_load_csr(g.n, rp, col, w)
    dev = [None if x is None else torch.from_numpy(x).cuda() for x in (rp, col, w)]
    got2, gid2 = ctx.try_load_csr(g.n, *dev)
    assert got == got2 == want
    assert (want == 0) == (kind == "whole")
    for i in (gid, gid2):
        if i >= 0:
            ctx.free_graph(i)
