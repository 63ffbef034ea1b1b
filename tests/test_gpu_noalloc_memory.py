"""ctb_contract_noalloc takes no device memory after the first call on a device,
whatever the shapes: the contraction has a kernel for each tile side, chunk
length and way of copying, and a kernel that is loaded on its first use takes
device memory then.  Run in a process of its own, where no other test has
loaded them."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
import torch
from paper_2604_08855_gb300 import build
build.build()
from paper_2604_08855_gb300 import ctb
shapes = [(1, 0), (5, 3), (8, 3), (8, 10), (10, 2), (10, 10), (10, 20), (16, 3), (16, 10), (16, 16), (20, 10), (24, 15),
          (36, 3), (36, 10), (40, 9), (64, 3), (20, 7), (32, 7), (6, 4), (6, 20), (32, 15), (28, 6), (12, 7), (7, 5)]
args = []
for nbins, lmax in shapes:
    a = torch.ones((64, nbins, (lmax + 1) ** 2 + 1), device="cuda")
    rows = a.view(-1)[: 64 * nbins * (lmax + 1) ** 2].view(64, nbins, (lmax + 1) ** 2)
    odd = a.view(-1)[1: 1 + rows.numel()].view_as(rows)  # rows that do not start on 16 bytes
    out = torch.empty((lmax + 1, nbins, nbins), device="cuda", dtype=torch.float64)
    args += [(rows, nbins, lmax, out), (odd, nbins, lmax, out)]
w = torch.ones(64, device="cuda")
ctb.contract_noalloc(args[0][0], w, *args[0][1:])
torch.cuda.synchronize()
free = torch.cuda.mem_get_info()[0]
for rows, nbins, lmax, out in args:
    ctb.contract_noalloc(rows, w, nbins, lmax, out)
torch.cuda.synchronize()
print("TAKEN", free - torch.cuda.mem_get_info()[0])
"""


def test_no_device_memory_for_further_shapes():
    pytest.importorskip("torch")
    r = subprocess.run([sys.executable, "-c", PROGRAM], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr
    assert r.stdout.split("TAKEN")[1].split() == ["0"]
