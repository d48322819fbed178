"""GPU: the status of a bad graph is that of its first failing category, wherever
the faults lie and however the blocks of the checks are scheduled.

The rows are many more than the check's warps, the fault of the earlier row is
of the later category, and other work on the GPU keeps some of the blocks from
starting until others have finished."""
import numpy as np
import pytest

from test_gpu_parity import ctx  # noqa: F401

pytestmark = pytest.mark.gpu

N = 200_003


def ring():
    """Every node joined to the next two."""
    u = np.arange(N)
    nb = np.sort(np.stack([(u - 2) % N, (u - 1) % N, (u + 1) % N, (u + 2) % N], 1), 1).astype(np.int32)
    return np.arange(N + 1, dtype=np.int64) * 4, nb.ravel(), np.ones(4 * N, np.float32)


def swap(col, e):
    col[e], col[e + 1] = col[e + 1], col[e]


def fault(kind, rp, col, w, u):
    """Give row u a fault of this category."""
    e = 4 * u
    if kind == "column":
        col[e] = N
    elif kind == "weight":
        w[e] = -1.0
    elif kind == "self-loop":
        col[e + 1] = u
    elif kind == "unsorted":
        swap(col, e)
    elif kind == "repeat":
        col[e] = col[e + 1]
    elif kind == "partner":
        w[e] = 2.0


@pytest.mark.parametrize("later,earlier", [("partner", "weight"), ("partner", "column"), ("repeat", "self-loop"),
                                           ("unsorted", "weight"), ("weight", "column"), ("partner", "repeat")])
@pytest.mark.parametrize("rows", [(0, N - 1), (N - 1, 0), (9727, 9728)])
def test_first_category(orc, ctx, later, earlier, rows):
    import torch

    rp, col, w = ring()
    fault(later, rp, col, w, rows[0])
    fault(earlier, rp, col, w, rows[1])
    want = orc.Graph(N, rp, col, w).status
    assert want != 0
    dev = [torch.from_numpy(x).cuda() for x in (rp, col, w)]
    a = torch.ones(4096, 4096, dtype=torch.bfloat16, device="cuda")
    b = torch.empty_like(a)
    torch.cuda.synchronize()
    side = torch.cuda.Stream()
    for _ in range(4):
        with torch.cuda.stream(side):
            for _ in range(12):
                torch.mm(a, a, out=b)
        got, gid = ctx.try_load_csr(N, *dev)
        assert (got, gid) == (want, -1)
    torch.cuda.synchronize()
