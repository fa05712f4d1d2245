"""Device memory of calls whose kernels could make the driver reserve local memory for every thread the GPU can hold:
measured in a process of its own, the context and the library's buffers included."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

HEAD = """
import torch
import paper_2210_11122_gb300 as mg
torch.zeros(1, device="cuda")
torch.cuda.synchronize()
free = torch.cuda.mem_get_info()[0]
"""
TAIL = """
torch.cuda.synchronize()
print("used_mib", (free - torch.cuda.mem_get_info()[0]) >> 20)
"""
SERVE = """
srv = mg.Server(slots=1, max_nevt=1024)
srv.wait(srv.submit("ggttggg", 5, 1024))
"""
BATCH = """
jobs = [(mg.Context(p), n) for p, n in ((3, 64), (2, 100), (1, 33), (0, 5))]
jobs = [(c, torch.zeros(c.mom_count(n), dtype=torch.float64, device="cuda"), n,
         torch.zeros(n, dtype=torch.float64, device="cuda")) for c, n in jobs]
for c, mom, n, me in jobs:
    c.rambo(3, n, 1500.0, mom)
mg.sigmakin_batch(jobs)
"""
TUNE = """
mg.Context(3).autotune(mg.MG_FP64, nevt=64)
"""


# 2.7 GB measured, 14.7 GB with a kernel of 50 KB of local memory per thread; the bound is twice the former
@pytest.mark.parametrize("code,bound_mib", [(SERVE, 5500), (BATCH, 5500), (TUNE, 5500)], ids=["server", "batch", "autotune"])
def test_device_memory(code, bound_mib):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    r = subprocess.run([sys.executable, "-c", HEAD + code + TAIL], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
    assert int(r.stdout.split("used_mib")[1]) <= bound_mib, r.stdout
