"""The memory of an instance whose 16-bit distances cannot be used."""
import os
import subprocess
import sys

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


CHILD = """
import sys, torch
from paper_1610_10061_gb300 import pm
torch.cuda.set_device(0)
d = torch.randint(0, 60000, (6000, 6000), device="cuda", dtype=torch.int32)
big = d.clone(); big[5999, 17] = 65536
many = d.clone(); many[:, 3] = 1 << 20
for x in (d, big, many):  # kernels are loaded once
    pm.Instance(x[:64, :64].contiguous(), 3).close()
    pm.Instance(x, 6).close()
for x in (d, big, many):
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    inst = pm.Instance(x, 6)
    torch.cuda.synchronize()
    print(before - torch.cuda.mem_get_info()[0])
    inst.close()
"""


def test_unused_entries_are_given_back():
    """In a child process without the memory pool, where free memory shows what an instance holds."""
    from paper_1610_10061_gb300 import build
    build.build()
    env = dict(os.environ, PM_POOL="0", PYTHONPATH=ROOT)
    out = subprocess.run([sys.executable, "-c", CHILD], capture_output=True, text=True, env=env, cwd=ROOT, timeout=300)
    assert out.returncode == 0, out.stderr
    fits, one, many = (int(v) for v in out.stdout.split())
    tables, entries, slack = 6000 * 6016 * 6, 750 * 6000 * 16, 8 << 20
    assert abs(fits - tables - entries) < slack
    assert abs(one - tables) < slack and abs(many - tables) < slack, (one, many)
