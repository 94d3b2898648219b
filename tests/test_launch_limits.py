"""A process that meets many sizes: after several hundred launch shapes, two
threads step meshes through one kernel at two shared-memory sizes, each on its
own stream, and no call may fail or spoil the other's result.  In a child
process, whose launch state starts empty.  GPU only."""
import os
import subprocess
import sys

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r"""
import threading
import torch
from paper_2201_03950_gb300 import trid

# strided FP64 systems of every height: one launch shape each, stored and added
nsys = 5000
for n in range(1, 257):
    t = [torch.full((nsys * n,), v, dtype=torch.float64, device="cuda")
         for v in (-1.0, 4.0, -1.0, 2.0)]
    trid.solve(*t, (nsys, n), 1, u=torch.zeros_like(t[3]))
    trid.solve(*t, (nsys, n), 1)

errors, results = [], {}

def step(name, dims, steps, calls):
    try:
        with torch.cuda.stream(torch.cuda.Stream()):
            u0 = torch.rand(dims[0] * dims[1] * dims[2], device="cuda")
            ws = torch.empty(trid.adi_workspace_bytes(dims, u0.dtype), dtype=torch.uint8,
                             device="cuda")
            for _ in range(calls):
                u = u0.clone()
                trid.adi_step(u, dims, 0.3, steps, ws)
            torch.cuda.current_stream().synchronize()
            results[name] = (u0, u, dims, steps)
    except Exception as e:
        errors.append((name, repr(e)))

threads = [threading.Thread(target=step, args=("large", (127, 126, 12), 200, 40)),
           threading.Thread(target=step, args=("small", (127, 101, 12), 1, 4000))]
for t in threads:
    t.start()
for t in threads:
    t.join()
assert not errors, errors
for u0, u, dims, steps in results.values():      # the same steps, undisturbed
    ws = torch.empty(trid.adi_workspace_bytes(dims, u.dtype), dtype=torch.uint8, device="cuda")
    assert torch.equal(trid.adi_step(u0, dims, 0.3, steps, ws), u)
print("ok")
"""


def test_two_sizes_of_one_kernel_after_many_shapes():
    r = subprocess.run([sys.executable, "-c", CHILD], cwd=ROOT, capture_output=True, text=True,
                       timeout=300)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stdout + r.stderr
