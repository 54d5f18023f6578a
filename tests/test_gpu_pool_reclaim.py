"""What the workspace pool keeps is there for an allocation that does not fit
without it, and comes back when the last state handle is freed.  In a process of
its own: other tests' handles would keep the memory."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SERVES = """
import torch, paper_0902_0699_gb300 as qc
s = qc.State(25, 0)  # 512 MiB; the sampler's CDF takes 256 MiB
s.uniform()
s.sample(1, 1 << 21)
torch.cuda.synchronize()
torch.cuda.empty_cache()
fill = torch.empty(torch.cuda.mem_get_info()[0] - (400 << 20), dtype=torch.uint8, device="cuda")
assert torch.cuda.mem_get_info()[0] < 512 << 20
qc.qc_state_free(qc.qc_state_alloc(25, 0))
"""

RETURNS = """
import torch, paper_0902_0699_gb300 as qc
s = qc.State(24, 0)
s.uniform()
s.sample(1, 1 << 20)
torch.cuda.synchronize()
before = torch.cuda.mem_get_info()[0]
s.close()
assert torch.cuda.mem_get_info()[0] >= before + (128 << 20)
"""


@pytest.mark.parametrize("code", [SERVES, RETURNS], ids=["serves an allocation", "comes back with the last handle"])
def test_kept_memory(code):
    r = subprocess.run([sys.executable, "-c", code], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr
