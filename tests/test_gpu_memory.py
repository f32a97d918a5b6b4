"""Device memory: what a domain takes beyond its vectors is given back when a call needs it."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

pytest.importorskip("paper_2111_06767_gb300")

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

_SCRIPT = r"""
import ctypes as C, os, sys, torch
sys.path.insert(0, sys.argv[1]); sys.path.insert(0, sys.argv[1] + "/tests")
import paper_2111_06767_gb300 as dgg
from paper_2111_06767_gb300 import _native as nat
from gpu_util import rand, rel

def held(d):
    lay = nat.dg_layout()
    assert dgg._lib.dg_domain_layout(d._h, C.byref(lay)) == nat.DG_OK
    return int(lay.device_bytes)

n, N = (4, 4, 4), 6
b = torch.from_numpy(rand(940, (64 * N**3,))).cuda()
u = torch.zeros_like(b)
d = dgg.Domain(n=n, N=N)
z = d.vcycle(b)                                          # the inverses, their digits, the work vectors
before = held(d)
os.environ["DG_ALLOC_LIMIT"] = str(before + (1 << 20))   # no room for a Krylov basis beside them
rep = d.solve(b, u, tol=1e-10)
assert rep.relative_residual <= 1e-10
print("held", before, held(d))
os.environ["DG_ALLOC_LIMIT"] = str(held(d) + (2 << 20))
for _ in range(3):                                       # host-driven, captured, replayed
    u.zero_()
    assert d.solve(b, u, tol=1e-10).relative_residual <= 1e-10
os.environ["DG_ALLOC_LIMIT"] = "1000000"                 # nothing left to give: an error, and the library goes on
try:
    dgg.Domain(n=n, N=N)
    raise SystemExit("no error")
except nat.NativeError as e:
    assert e.status == -2, e
del os.environ["DG_ALLOC_LIMIT"]
ref = torch.zeros_like(b)
s = dgg.Domain(n=n, N=N, gemm="simt")
assert s.solve(b, ref, tol=1e-10).iterations == rep.iterations
assert rel(u.cpu().numpy(), ref.cpu().numpy()) < 1e-9
assert rel(d.vcycle(b).cpu().numpy(), z.cpu().numpy()) < 1e-12
"""


def test_a_solve_that_needs_the_memory_gets_that_of_the_digit_slices(tmp_path):
    """An FP64 domain whose digit slices leave no room for the Krylov basis solves with the CUDA-core product instead of
    ending out of memory (DG_ALLOC_LIMIT stands in for the device's size): one solve, then captured and replayed ones."""
    f = tmp_path / "run.py"
    f.write_text(_SCRIPT)
    r = subprocess.run([sys.executable, str(f), ROOT], timeout=600, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
