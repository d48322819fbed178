"""GPU: initial communities that each share nodes with as many others as a warp's
table of partners holds (512 of 1,024 entries), and more: the full method against
the oracle."""
import numpy as np
import pytest

from paper_1301_0955_gb300 import synth
from test_gpu_full import compare, ctx  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("met", [511, 512, 513, 640, 1024, 1500])
def test_few_members_many_partners(orc, ctx, met):
    g = synth.config_graph(0)
    r = np.random.default_rng(met)
    # every community holds one of two nodes that stand first, and others of its own
    lists = [np.concatenate([[7, 450], r.choice(np.setdiff1d(np.arange(g.n), [7, 450]), 5 + i % 4, replace=False)])
             for i in range(met + 1)]
    ptr = np.concatenate([[0], np.cumsum([len(x) for x in lists])]).astype(np.int64)
    compare(orc, ctx, g, np.array([3.0]), init=(ptr, np.concatenate(lists).astype(np.int32)), eta=0.95)
