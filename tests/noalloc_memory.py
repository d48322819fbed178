"""Child process of test_gpu_noalloc_memory.py: the device's free memory across
calls of mscd_grow_noalloc, after one call on a small graph."""
import json
import os
import sys

import numpy as np
import torch

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
from paper_1301_0955_gb300 import mscd, synth  # noqa: E402


def star(leaves, weighted, more=0):
    """A centre with `leaves` leaves, and one with `more` apart from it."""
    u = np.concatenate([np.zeros(leaves, np.int64), np.full(more, leaves + 1, np.int64)])
    v = np.concatenate([np.arange(1, leaves + 1), leaves + 1 + np.arange(1, more + 1)])
    n = leaves + 1 + (more + 1 if more else 0)
    return n, *synth.to_csr(n, u, v, np.ones(len(u), np.float32) if weighted else None)


def outputs(U, need):
    z = dict(device="cuda:0")
    return dict(nodes=torch.zeros(need, dtype=torch.int32, **z), offset=torch.zeros(U, dtype=torch.int64, **z),
                len=torch.zeros(U, dtype=torch.int32, **z), fitness=torch.zeros(U, dtype=torch.float64, **z),
                stats=torch.zeros((U, mscd.NSTATS), dtype=torch.int64, **z),
                status=torch.zeros(U, dtype=torch.int32, **z), hash=torch.zeros(U, dtype=torch.int64, **z))


ctx = mscd.Context(0)
# 6,000 leaves outgrow the shared-memory classes; a centre of 33,000 takes the
# wider unweighted slots, weights the widest
cases = {"15 bits": star(6000, False), "32 bits": star(6000, False, 33_000), "weighted": star(6000, True)}
small = synth.config_graph(0)
gid0 = ctx.load_csr(small.n, small.row_ptr, small.col)
gids = {k: ctx.load_csr(*g) for k, g in cases.items()}
seeds = torch.arange(1, 41, dtype=torch.int32, device="cuda:0")
out0 = outputs(40, 1 << 16)
out = {k: outputs(40, 1 << 16) for k in cases}
torch.cuda.synchronize()
rc, _ = ctx.grow_noalloc(gid0, np.array([1.0]), seeds, out0)
assert rc == mscd.OK, rc
torch.cuda.synchronize()
report = {}
for k, gid in gids.items():
    before = torch.cuda.mem_get_info()[0]
    rc, _ = ctx.grow_noalloc(gid, np.array([450.0]), seeds, out[k])
    torch.cuda.synchronize()
    lens = out[k]["len"].cpu()
    report[k] = {"rc": rc, "taken": before - torch.cuda.mem_get_info()[0], "members": int(lens.min())}
print(json.dumps(report))
