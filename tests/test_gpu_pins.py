"""The switches that pin a launch shape (DG_GEMM_SPLIT, DG_APPLY_VARIANT) pin it: the tuner is not asked, and the
results are those of the pinned shape."""
import os
import subprocess
import sys

import numpy as np
import pytest
import torch

from gpu_util import rand

pytestmark = pytest.mark.gpu

dgg = pytest.importorskip("paper_2111_06767_gb300")

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.mark.parametrize("n,N,ov", [((2, 1, 1), 6, 2), ((5, 4, 3), 6, 2), ((3, 3, 3), 8, 2)])
def test_the_fp64_product_does_not_depend_on_its_k_split(monkeypatch, n, N, ov):
    """The digits' sums are integers: 1, 2, 4 or 8 CTAs per tile (11 and 20 K chunks, uneven shares) give the same bits."""
    m = n[0] * n[1] * n[2] * N**3
    b, u = (torch.from_numpy(rand(s, (m,))).cuda() for s in (930, 931))
    out = {}
    for split in (1, 2, 4, 8):
        monkeypatch.setenv("DG_GEMM_SPLIT", str(split))
        d = dgg.Domain(n=n, N=N, mg_levels=1, overlap=ov, neumann=(1,))
        out[split] = d.schwarz_smooth(0, b, u.clone(), 2).cpu().numpy()
    assert all(np.array_equal(out[1], out[s]) for s in (2, 4, 8))


def _log_of(script, tmp_path, **env):
    f = tmp_path / "run.py"
    f.write_text("import sys, torch\nsys.path.insert(0, %r)\nimport paper_2111_06767_gb300 as dgg\n" % ROOT + script)
    r = subprocess.run([sys.executable, str(f)], env=dict(os.environ, DG_TUNE_LOG="1", **env), check=True, timeout=600,
                       capture_output=True, text=True)
    return r.stderr


_SMOOTH = """
for prec, gemm in (("fp64", "default"), ("fp64", "simt"), ("mixed", "tf32")):
    d = dgg.Domain(n=(4, 4, 4), N=6, mg_levels=1, overlap=2, precision=prec, gemm=gemm)
    b = torch.ones(d.n_dof, dtype=torch.float64, device="cuda")
    d.schwarz_smooth(0, b, torch.zeros_like(b), 1)
"""


@pytest.mark.parametrize("split", ["1", "4"])
def test_a_pinned_gemm_split_is_not_tuned(tmp_path, split):
    log = _log_of(_SMOOTH, tmp_path, DG_GEMM_SPLIT=split)
    assert "dg autotune key 1 " in log  # the applies are tuned
    for key in (3, 4, 5):  # the tensor-core products and the CUDA-core one are not
        assert f"dg autotune key {key} " not in log


_APPLY = """
for N in (4, 7):
    d = dgg.Domain(n=(3, 2, 2), N=N, mg_levels=1, overlap=2)
    u = torch.ones(d.n_dof, dtype=torch.float64, device="cuda")
    d.apply(u)
    d.apply_f32(u.float())
    d.schwarz_smooth(0, u, u.clone(), 1)
"""


@pytest.mark.parametrize("variant", ["0", "1", "2", "3", "4"])
def test_a_pinned_apply_shape_is_not_tuned(tmp_path, variant):
    """Also where the grid is too small for the tuner to be offered the shape."""
    assert "dg autotune key 1 " not in _log_of(_APPLY, tmp_path, DG_APPLY_VARIANT=variant)


def test_a_shape_that_does_not_exist_is_reported_and_tuned(tmp_path):
    log = _log_of(_APPLY, tmp_path, DG_APPLY_VARIANT="5")
    assert log.count("dg DG_APPLY_VARIANT=5: no such launch shape here") == 1 and "dg autotune key 1 " in log
