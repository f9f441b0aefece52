"""Device memory that a build takes, scratch included, in a process of its own."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = """
import torch
from paper_1902_08083_gb300 import trevr
n, s = 1 << 22, 1 << 14
a = [torch.rand(3, n, device="cuda"), torch.rand(n, device="cuda"),
     torch.rand(3, s, device="cuda"), torch.rand(s, device="cuda")]
few = [a[0][:, :64].contiguous(), a[1][:64].contiguous(), a[2], a[3]]
trevr.build_tree(*few)  # the pool, and what the kernels need
torch.cuda.synchronize()
before = torch.cuda.mem_get_info()[0]
t = trevr.build_tree(*a)
print((before - torch.cuda.mem_get_info()[0]) / n, t.n_nodes / n)
"""


def test_a_build_takes_at_most_200_bytes_a_particle():
    # 78 for the particles, in order and while they are sorted, and 276 for a cell, of which
    # there are 0.36 per particle, and its sums; the pool grows in steps of 32 MB (8 each)
    r = subprocess.run([sys.executable, "-c", PROGRAM], cwd=ROOT, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    per, cells = (float(x) for x in r.stdout.split())
    assert 78 + 276 * cells < 180
    assert per < 200, per
