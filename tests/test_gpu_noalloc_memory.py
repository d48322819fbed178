"""GPU: after its first call on a device, mscd_grow_noalloc takes no device memory,
whichever of its kernels a later call is the first to need."""
import json
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu


def test_free_memory_after_a_small_first_call():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1301_0955_gb300 import build

    build.build()
    # a process of its own: what other tests have run is loaded already
    child = os.path.join(os.path.dirname(os.path.abspath(__file__)), "noalloc_memory.py")
    p = subprocess.run([sys.executable, child], capture_output=True, text=True, timeout=300)
    assert p.returncode == 0, p.stderr
    report = json.loads(p.stdout.strip().splitlines()[-1])
    assert set(report) == {"15 bits", "32 bits", "weighted"}
    for k, r in report.items():
        assert r["rc"] == 0 and r["members"] > 2, (k, r)
        assert r["taken"] == 0, report
