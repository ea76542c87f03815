"""A reduction on a device with little memory left: when the arena cannot grow any
more, fewer columns are reduced at a time, and the bars are the same.  In a
process of its own, so that no earlier call has left a larger arena."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

CHILD = """
import sys
import numpy as np, torch
import oracle
import paper_1908_02518_gb300 as rg
oracle.build()
a = np.tril(np.random.Generator(np.random.PCG64(200)).random((200, 200)).astype(np.float32), -1)
d = a + a.T
key = lambda bars: sorted((int(b["dim"]), float(b["birth"]), float(b["death"]), int(b["birth_simplex"]),
                           int(b["death_simplex"]) % 2**64) for b in bars)
want = key(oracle.barcodes(d, 1).bars)
x = torch.from_numpy(d).cuda()
rg.barcodes(x[:50, :50].contiguous(), 1)  # the library is loaded and its small buffers are there
left = int(float(sys.argv[1]) * 2**30)
held = torch.empty(torch.cuda.mem_get_info()[0] - left, dtype=torch.uint8, device="cuda")
assert key(rg.barcodes(x, 1).bars) == want
print("ok")
"""


@pytest.mark.parametrize("gigabytes", [8, 2])
def test_fewer_columns_at_a_time_when_memory_is_short(gigabytes):
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", CHILD, str(gigabytes)], cwd=root, capture_output=True, text=True,
                       timeout=300)
    assert r.returncode == 0 and "ok" in r.stdout, r.stderr[-2000:]
