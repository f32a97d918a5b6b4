"""Every launch shape of the direction-by-direction DG apply against the oracle, at every order.

Each shape (few / middle / many elements per CTA, the three directions side by side) is pinned for a
process of its own and runs the operator on grids whose element counts no brick divides, on a single
element and with Neumann faces, in FP64 (1e-12 relative) and FP32 (2e-5, as the other operator
tests), and the residual written into the subdomain vectors through two FP64 Schwarz steps (1e-10,
as the other smoother tests).
"""
import functools
import os
import subprocess
import sys

import numpy as np
import pytest

from gpu_util import rand, rel
from oracle import dg, schwarz

pytestmark = pytest.mark.gpu

GRIDS = [((1, 1, 1), ()), ((3, 2, 1), (5,)), ((5, 3, 4), (0, 2)), ((17, 1, 2), (1, 4))]
LOWER, UPPER = (-1.0, -0.5, 0.0), (1.0, 0.7, 2.5)

_SCRIPT = r"""
import sys, numpy as np, torch
sys.path.insert(0, sys.argv[2]); sys.path.insert(0, sys.argv[2] + "/tests")
import paper_2111_06767_gb300 as dgg
from gpu_util import rand
from test_gpu_dir_apply import GRIDS, LOWER, UPPER
out = {}
for N in range(2, 11):
    for c, (n, neu) in enumerate(GRIDS):
        d = dgg.Domain(LOWER, UPPER, n, N, mg_levels=1, overlap=1, neumann=neu)
        u = torch.from_numpy(rand(700 + c, (n[0] * n[1] * n[2], N, N, N)).ravel()).cuda()
        out[f"f64_{N}_{c}"] = d.apply(u).cpu().numpy()
        out[f"f32_{N}_{c}"] = d.apply_f32(u.float()).double().cpu().numpy()
    n = (3, 2, 2)
    d = dgg.Domain(n=n, N=N, mg_levels=1, overlap=min(2, N - 1), neumann=(3,))
    b, u = (torch.from_numpy(rand(s, (12, N, N, N)).ravel()).cuda() for s in (801, 802))
    out[f"smooth_{N}"] = d.schwarz_smooth(0, b, u, 2).cpu().numpy()
np.savez(sys.argv[1], **out)
"""


@functools.cache
def _references():
    ref = {}
    for N in range(2, 11):
        for c, (n, neu) in enumerate(GRIDS):
            grid = dg.BoxGrid(LOWER, UPPER, n, N, 1.5, tuple(fc in neu for fc in range(6)))
            ref[f"{N}_{c}"] = dg.apply(grid.graph(), rand(700 + c, (grid.n_elements, N, N, N)))
        grid = dg.BoxGrid((-1.0,) * 3, (1.0,) * 3, (3, 2, 2), N, 1.5, tuple(fc == 3 for fc in range(6)))
        b, u = (rand(s, (12, N, N, N)) for s in (801, 802))
        ref[f"smooth_{N}"] = schwarz.SchwarzLevel(grid, min(2, N - 1)).smooth(b, u, 2)
    return ref


@pytest.mark.parametrize("variant", ["1", "2", "3", "4"])
def test_every_launch_shape_matches_oracle(tmp_path, variant):
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    script, f = tmp_path / "run.py", tmp_path / "out.npz"
    script.write_text(_SCRIPT)
    subprocess.run([sys.executable, str(script), str(f), root], env=dict(os.environ, DG_APPLY_VARIANT=variant),
                   check=True, timeout=600)
    got, ref = np.load(f), _references()
    for N in range(2, 11):
        for c in range(len(GRIDS)):
            assert rel(got[f"f64_{N}_{c}"], ref[f"{N}_{c}"]) < 1e-12, (N, c)
            assert rel(got[f"f32_{N}_{c}"], ref[f"{N}_{c}"]) < 2e-5, (N, c)
        assert rel(got[f"smooth_{N}"], ref[f"smooth_{N}"]) < 1e-10, N
