"""csr_encode_static takes device memory at the first call for a dictionary shape only, whatever the numbers of rows
of the calls that follow (each of them may launch other kernels).  In a process of its own: the
runtime loads a kernel's code once per process."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r'''
import sys
import torch
sys.path.insert(0, %(root)r)
import paper_2412_11741_b200 as csr
dev, N, d, s = "cuda:0", %(N)d, %(d)d, 4
D = torch.nn.functional.normalize(torch.randn(N, d, device=dev), dim=1).contiguous()
X = torch.randn(60000, d, device=dev).to(torch.bfloat16)
oi = torch.zeros((60000, s), dtype=torch.int16, device=dev).view(torch.uint16)
oc = torch.zeros((60000, s), dtype=torch.float16, device=dev)
status = torch.zeros(1, dtype=torch.int32, device=dev)
rows = (%(first)d, 1, 8, 100, 1500, 12000, 18945, 37888, 60000)
free = []
for M in rows:
    csr.csr_encode_static(D, X[:M], s, oi[:M], oc[:M], dev_status=status)
    torch.cuda.synchronize()
    free.append(torch.cuda.mem_get_info()[0])
print("FREE", free[0], min(free[1:]))
'''


@pytest.mark.parametrize("N,d,first", [(4096, 128, 16), (4096, 128, 60000), (3000, 64, 60000)])
def test_calls_after_the_first_take_no_device_memory(N, d, first):
    from paper_2412_11741_b200 import build
    build.build()
    res = subprocess.run([sys.executable, "-c", CHILD % {"root": ROOT, "N": N, "d": d, "first": first}], capture_output=True, text=True, timeout=600)
    assert res.returncode == 0, res.stdout + res.stderr
    after_first, least = (int(v) for v in [l for l in res.stdout.splitlines() if l.startswith("FREE")][0].split()[1:])
    assert least == after_first, (after_first, least)
