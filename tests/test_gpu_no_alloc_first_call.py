"""recon_gram_inverse_noalloc takes device memory in its first call on a device only, whichever of its two
forms (tensor cores, FP64) that call takes: each order in a process of its own, so that nothing else has
loaded the kernels of the other form."""

import os
import subprocess
import sys

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = """
import sys
import torch
from paper_1203_4587_gb300 import binding
sizes = [(int(s.split(":")[0]), float(s.split(":")[1])) for s in sys.argv[1:]]
args = []
for n, mu in sizes:
    mask = (torch.arange(n, device="cuda") % 3 == 0).to(torch.uint8).repeat(200, 1)
    sens = torch.full((200, 2, n), 0.7, dtype=torch.complex64, device="cuda")
    args.append((mask, sens, mu, torch.empty((200, n, n), dtype=torch.complex64, device="cuda")))
binding.load()
free = []
for mask, sens, mu, out in args:
    binding.gram_inverse_noalloc(mask, sens, mu, out=out)
    torch.cuda.synchronize()
    free.append(torch.cuda.mem_get_info()[0])
print(free)
sys.exit(0 if min(free) == max(free) else 1)
"""


# blocks of 16 and an ill-conditioned 64 in FP64; 40, 64 and 160 on the tensor cores (one and several waves)
@pytest.mark.parametrize("order", [("16:0.1", "64:0.1", "160:0.1", "40:0.1"), ("160:0.1", "64:0.1", "16:0.1"),
                                   ("64:0.001", "160:0.1", "64:0.1")])
def test_later_calls_take_no_device_memory(order):
    r = subprocess.run([sys.executable, "-c", PROGRAM, *order], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, (r.stdout, r.stderr[-2000:])
