"""The scratch pool gives its memory back with the device's last grid and batch, also when the last
one is a batch whose scratch is freed in stream order.  In a process of its own: other tests' grids
would keep the pool."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CODE = """
import torch
from paper_2404_10272_gb300 import hdda as H
n = 1 << 20
o = torch.zeros((n, 3), device="cuda")
d = torch.ones((n, 3), device="cuda")
occ = torch.ones((1, 16, 16, 16), dtype=torch.uint8, device="cuda")
grid = H.build_vdb(occ, [[-1, -1, -1, 1, 1, 1]])
out = H.alloc_samples(n, 1)
job = dict(rays_o=o, rays_d=d, grid=grid, params=H.make_params(0.0, 0.5, 0.1), out=out)
for last in ("batch", "grid"):
    grid = H.build_vdb(occ, [[-1, -1, -1, 1, 1, 1]])
    batch = H.Batch([dict(job, grid=grid)], use_graph=False)
    batch.launch()
    torch.cuda.synchronize()
    job["grid"].free()
    if last == "batch":
        grid.free()  # nothing is launched any more
    held = torch.cuda.mem_get_info()[0]
    batch.free()
    grid.free()
    torch.cuda.synchronize()
    print(last, (torch.cuda.mem_get_info()[0] - held) >> 20)
"""


def test_memory_goes_back():
    r = subprocess.run([sys.executable, "-c", CODE], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
    got = dict(line.split() for line in r.stdout.splitlines())
    # the batch's scratch is 134 bytes per ray: 134 MiB
    assert int(got["batch"]) >= 128 and int(got["grid"]) >= 128, got
