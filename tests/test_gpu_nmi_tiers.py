"""GPU: the NMI's tiers (a warp, a CTA, a global table per community) and its
terms with and without the table, against the oracle."""
import numpy as np
import pytest

from test_gpu_nmi import ctx  # noqa: F401

pytestmark = pytest.mark.gpu


def cover(lists):
    ptr = np.concatenate([[0], np.cumsum([len(x) for x in lists])]).astype(np.int64)
    return ptr, np.concatenate(lists).astype(np.int32)


def pick(rng, n, m):
    return np.sort(rng.choice(n, m, replace=False))


CASES = {
    # partners met by one community of the first cover: below and above a warp's 256
    "256 partners": lambda r: (4000, [np.arange(2000)], [pick(r, 4000, 9) for _ in range(256)]),
    "600 partners": lambda r: (4000, [np.arange(2000), pick(r, 4000, 40)], [pick(r, 4000, 9) for _ in range(600)]),
    # few partners, more list entries than a warp walks (16,384)
    "many entries": lambda r: (4000, [np.arange(0, 4000, 2), pick(r, 4000, 31)],
                               [pick(r, 4000, 3000) for _ in range(20)]),
    # above a CTA's 4,096: the global table; large disjoint partners among them
    "5000 partners": lambda r: (9000, [np.arange(5000), np.arange(5000, 9000), pick(r, 9000, 33)],
                                [np.array([i, 8999 - i // 4]) for i in range(5000)] + [np.arange(5000, 9000)[1:]]),
    # more nodes than the terms are tabled for
    "2^26 nodes": lambda r: (2 ** 26 + 5, [pick(r, 10 ** 6, 500) for _ in range(3)],
                             [pick(r, 10 ** 6, 400) for _ in range(3)] + [np.arange(100)]),
}


@pytest.mark.parametrize("name", list(CASES))
def test_tiers(orc, ctx, name):
    n, a, b = CASES[name](np.random.default_rng(3))
    a, b = cover(a), cover(b)
    want = orc.nmi(n, a[0], a[1], b[0], b[1])
    assert ctx.nmi_covers(n, a, b) == pytest.approx(want, abs=1e-12)
    assert ctx.nmi_covers(n, b, a) == pytest.approx(want, abs=1e-12)
