"""GPU: the volume's limit of 2^62 units, where the sum is made (within a row's
lanes, over rows, warps and blocks), and sums that would wrap around 64 bits to
something small.  Statuses, degrees and volumes against the oracle's."""
import numpy as np
import pytest

from paper_1301_0955_gb300 import synth
from test_gpu_parity import ctx  # noqa: F401

pytestmark = pytest.mark.gpu


def edges(where, heavy):
    """`heavy` node pairs: of one row, of rows next to each other, or of far rows."""
    i = np.arange(heavy)
    if where == "row":
        return 70, np.zeros(heavy, np.int64), 1 + i
    if where == "rows":
        return 70, 2 * i, 2 * i + 1
    return 400_001, 2 * (i * 6_200), 2 * (i * 6_200) + 1


@pytest.mark.parametrize("where", ["row", "rows", "far rows"])
@pytest.mark.parametrize("log2_w,heavy", [(60, 1), (60, 2), (61, 1), (62, 1), (63, 1), (59, 3), (59, 4), (60, 4), (60, 8),
                                          (60, 16), (58, 32), (58, 7), (58, 8)])
def test_volume_limit(orc, ctx, where, log2_w, heavy):
    n, u, v = edges(where, heavy)
    # one pair of weight 1 fixes the unit, and is what is left of a sum that wraps
    u, v = np.append(u, n - 2), np.append(v, n - 1)
    w = np.append(np.full(heavy, 2.0 ** log2_w), 1.0).astype(np.float32)
    rp, col, ww = synth.to_csr(n, u, v, w)
    G = orc.Graph(n, rp, col, ww)
    got, gid = ctx.try_load_csr(n, rp, col, ww)
    volume = heavy * 2 ** (log2_w + 1) + 2
    assert got == G.status and (got == 0) == (volume < 2 ** 62)
    if gid >= 0:
        k = ctx.graph_degrees(gid)
        assert sum(int(x) for x in k) == volume
        assert k[n - 1] == 1 and int(k.max()) == 2 ** log2_w * (heavy if where == "row" else 1)
        ctx.free_graph(gid)
