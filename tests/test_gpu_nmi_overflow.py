"""GPU: communities whose partners overflow a CTA's count table (4,096) while all
of its warps are still walking members, in turn with communities that fit the
table the first ones leave behind.  Against the oracle."""
import numpy as np
import pytest

from test_gpu_nmi import ctx  # noqa: F401
from test_gpu_nmi_tiers import cover, pick

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("partners,size", [(9000, 5), (20000, 4), (5200, 3)])
def test_table_overflow_amid_the_walk(orc, ctx, partners, size):
    r = np.random.default_rng(partners)
    n = 12000
    # 2,000 members overflow the table (in the third case some of 2,000, all of
    # 12,000 do), 700 fit it, 4 fit a warp's
    a = [np.arange(2000 * i, 2000 * (i + 1)) for i in range(6)]
    a += [pick(r, n, 700) for _ in range(40)] + [pick(r, n, 2000) for _ in range(12)] + [pick(r, n, 4)]
    a += [np.arange(n)]
    b = [pick(r, n, size) for _ in range(partners)]
    a, b = cover(a), cover(b)
    want = orc.nmi(n, a[0], a[1], b[0], b[1])
    for _ in range(3):
        assert ctx.nmi_covers(n, a, b) == pytest.approx(want, abs=1e-12)
    assert ctx.nmi_covers(n, b, a) == pytest.approx(want, abs=1e-12)


@pytest.mark.parametrize("met", [255, 256, 257, 384, 512, 700])
def test_few_members_many_partners(orc, ctx, met):
    """Communities of 11 members that all lie in the same `met` partners: a warp's
    table (512 entries, listed up to 256) is at its limit before the first
    members have been walked, and what comes after must still be counted where it
    is not given up."""
    r = np.random.default_rng(met)
    n = 3000
    core = np.arange(40)
    a = [pick(r, 40, 11) for _ in range(60)] + [pick(r, n, 30) for _ in range(20)]
    b = [np.concatenate([core, 40 + pick(r, n - 40, 1 + i % 90)]) for i in range(met)]
    a, b = cover(a), cover(b)
    want = orc.nmi(n, a[0], a[1], b[0], b[1])
    assert ctx.nmi_covers(n, a, b) == pytest.approx(want, abs=1e-12)
    assert ctx.nmi_covers(n, b, a) == pytest.approx(want, abs=1e-12)


@pytest.mark.parametrize("lists", [63, 64, 65, 127, 128, 129])
def test_lists_about_the_line_between_the_walks(orc, ctx, lists):
    """Every node in exactly `lists` communities of the second cover (64 entries a
    list is the line, 128 a step); communities of 1 to 70 members, so that the last
    32 of them are fewer."""
    r = np.random.default_rng(lists)
    n = 480
    a = [pick(r, n, m) for m in (1, 2, 31, 32, 33, 63, 64, 65, 70)] + [pick(r, n, 200)]
    b = [p for _ in range(lists) for p in np.split(r.permutation(n), [40, 160, 170])]
    a, b = cover(a), cover([np.sort(x) for x in b])
    want = orc.nmi(n, a[0], a[1], b[0], b[1])
    assert ctx.nmi_covers(n, a, b) == pytest.approx(want, abs=1e-12)
    assert ctx.nmi_covers(n, b, a) == pytest.approx(want, abs=1e-12)
