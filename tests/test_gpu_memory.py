"""Device memory: what a domain takes beyond its vectors is given back when a call needs it, and the server admits a
request only where all that its domain will hold fits the budget."""
import ctypes as C
import os
import subprocess
import sys

import numpy as np
import pytest

import workloads
from gpu_util import rand

pytestmark = pytest.mark.gpu

dgg = pytest.importorskip("paper_2111_06767_gb300")
from paper_2111_06767_gb300 import _native as nat  # noqa: E402

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


_BATCH_SCRIPT = r"""
import ctypes as C, os, sys, torch
sys.path.insert(0, sys.argv[1]); sys.path.insert(0, sys.argv[1] + "/tests")
import paper_2111_06767_gb300 as dgg
from test_gpu_memory import _held
from gpu_util import rand, rel

shapes = [((8, 8, 8), 4), ((4, 4, 4), 6)]  # the first needs more than its own slices take, the second holds the larger ones
doms, bs, us, ref = [], [], [], []
for i, (n, N) in enumerate(shapes):
    d = dgg.Domain(n=n, N=N)
    b = torch.from_numpy(rand(941 + i, (d.n_dof,))).cuda()
    s = dgg.Domain(n=n, N=N, gemm="simt")
    r = torch.zeros_like(b)
    s.solve(b, r, tol=1e-10)
    ref.append(r.cpu().numpy())
    s.close()
    d.vcycle(b)
    doms.append(d); bs.append(b); us.append(torch.zeros_like(b))
os.environ["DG_ALLOC_LIMIT"] = str(sum(_held(d) for d in doms) + (1 << 20))
batch = dgg.Batch(doms, bs, us, tol=1e-10)
for r in batch.run():
    assert r.relative_residual <= 1e-10
for u, r in zip(us, ref):
    assert rel(u.cpu().numpy(), r) < 1e-9
"""


def test_a_batch_takes_the_memory_of_its_other_domains_slices(tmp_path):
    f = tmp_path / "run.py"
    f.write_text(_BATCH_SCRIPT)
    r = subprocess.run([sys.executable, str(f), ROOT], timeout=600, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]


def _held(d):
    lay = nat.dg_layout()
    assert dgg._lib.dg_domain_layout(d._h, C.byref(lay)) == nat.DG_OK
    return int(lay.device_bytes)


@pytest.mark.parametrize("kind,n,N,precision,max_it", [
    ("poisson", (24, 24, 24), 2, "mixed", 1), ("poisson", (24, 24, 24), 2, "fp64", 1), ("poisson", (9, 8, 7), 6, "mixed", 3),
    ("poisson", (6, 5, 4), 7, "fp64", 64), ("coef", (12, 12, 12), 2, "mixed", 2), ("coef", (4, 4, 4), 5, "fp64", 2),
    ("puncture", (8, 8, 8), 5, "mixed", 2), ("puncture", (4, 4, 4), 4, "fp64", 20)])
def test_a_budget_below_what_the_domain_holds_refuses_the_request(kind, n, N, precision, max_it):
    """The admission estimate is an upper bound: a domain that has solved as the server's do (three times, so that it
    holds the captured solve as well) holds no more, and a budget one byte below that is refused."""
    m = n[0] * n[1] * n[2] * N**3
    more = {}
    if kind == "coef":
        more["coef"] = 1.0 + 0.2 * rand(950, (m,))
    if kind == "puncture":
        more.update(problem="puncture", punctures=workloads.BINARY_PUNCTURES, lower=(-20.0,) * 3, upper=(20.0,) * 3)
    box = dict(lower=(-1.0,) * 3, upper=(1.0,) * 3)
    box.update(more)
    f = None if kind == "puncture" else rand(951, (m,))
    opts = dgg.solve_opts(max_iterations=max_it)
    overlap = min(2, N - 1)
    d = dgg.Domain(n=n, N=N, precision=precision, overlap=overlap, gemm="simt" if precision == "fp64" else "default", **box)
    for _ in range(3):
        try:
            d.solve_host(f, np.zeros(m), tol=1e-10, opts=opts)
        except nat.NativeError:
            pass  # so few iterations need not converge
    desc = dgg.make_desc(n=n, N=N, precision=precision, overlap=overlap, **box)
    srv = dgg.Server(max_active=1, n_streams=1, memory_budget_bytes=_held(d) - 1)
    try:
        with pytest.raises(nat.NativeError):
            srv.submit(desc, f, opts=opts)
    finally:
        srv.close()
