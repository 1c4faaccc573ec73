"""SSD workspace sizes of empty problems: zero heads, zero batch rows and zero
tokens are valid sizes, and every query answers them. Asked in a process of
their own, since a fault in the host code would end it."""

import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
QUERY = """
from paper_2607_02805_gb300 import binding as b
d = b.make_ssd_dims({batch}, {length}, {block}, {heads}, {n})
print(b.bdscan_ssd_forward_workspace_size(d), b.bdscan_ssd_boundary_states_workspace_size(d, 0),
      b.bdscan_ssd_boundary_states_workspace_size(d, 1), b.bdscan_ssd_full_bidir_workspace_size(d),
      b.bdscan_ssd_backward_workspace_size(d), repr(b.bdscan_last_error()))
"""


@pytest.mark.parametrize("batch,length,heads", [(2, 512, 0), (0, 512, 0), (2, 0, 0), (0, 512, 3), (2, 0, 3)])
@pytest.mark.parametrize("block,n", [(128, 64), (256, 128)])
def test_every_size_query_answers(batch, length, heads, block, n):
    src = QUERY.format(batch=batch, length=length, heads=heads, block=block, n=n)
    r = subprocess.run([sys.executable, "-c", src], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, (r.returncode, r.stderr[-500:])
    sizes = [int(v) for v in r.stdout.split()[:5]]
    assert all(0 <= v < 1 << 34 for v in sizes), r.stdout
