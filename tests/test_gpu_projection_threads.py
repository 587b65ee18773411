"""mcf_project_capped_simplex with its distance from threads that have not used the device before, in a
fresh process: as the process's first call into the library (which makes the memory pool), again
from another fresh thread, and from the main thread, with the same results."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = """
import threading, torch
from paper_2501_17996_gb300 import binding
g = torch.Generator(device="cuda").manual_seed(1)
n, m = 300, 2000
Q = torch.randn((m, n), device="cuda", generator=g)
cap = torch.rand(m, device="cuda", generator=g) + 0.1
torch.cuda.synchronize()
out = []
def project():
    F, mu = torch.empty_like(Q), torch.zeros(m, device="cuda")
    torch.cuda.synchronize()
    ptrs = Q.data_ptr(), cap.data_ptr(), F.data_ptr(), mu.data_ptr()
    box = []
    t = threading.Thread(target=lambda: box.append(binding.mcf_project_capped_simplex(n, m, n, *ptrs, 0)))
    t.start(); t.join()
    out.append((F, mu, box[0]))
project(); project()
F, mu = torch.empty_like(Q), torch.zeros(m, device="cuda")
d = binding.mcf_project_capped_simplex(n, m, n, Q.data_ptr(), cap.data_ptr(), F.data_ptr(), mu.data_ptr(), 0)
torch.cuda.synchronize()
for F2, mu2, d2 in out:
    assert torch.equal(F, F2) and torch.equal(mu, mu2) and d == d2
q64 = Q.double()
assert abs(float((F.double() - q64).square().sum()) - d) <= 1e-4 * d
print("same")
"""


def test_first_use_from_threads_without_a_context(lib):
    r = subprocess.run([sys.executable, "-c", PROGRAM], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.strip() == "same", r.stdout + r.stderr
