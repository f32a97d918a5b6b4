"""Rounding of the FP32 apply against the oracle's FP64 one, in units of FP32 rounding (2^-23)."""
import numpy as np
import pytest
import torch

from gpu_util import rand
from oracle import dg

pytestmark = pytest.mark.gpu

dgg = pytest.importorskip("paper_2111_06767_gb300")


@pytest.mark.parametrize("N", range(5, 11))
def test_fp32_apply_is_right_to_six_tenths_of_a_unit(N):
    """A result's own rounding is 0.29 units in norm; every sum, weight and flux before it adds some. Emulated with one
    rounding for the three weights together: 0.45-0.55 (rounded weights and products: 0.58-0.96)."""
    for n, upper in (((5, 4, 3), (1.0, 1.0, 1.0)), ((4, 5, 4), (1.0, 0.7, 2.5))):
        grid = dg.BoxGrid((-1.0, -0.5, 0.0), upper, n, N, 1.5, (False,) * 6)
        u = rand(960 + N, (grid.n_elements, N, N, N)).astype(np.float32)
        ref = dg.apply(grid.graph(), u.astype(np.float64))
        d = dgg.Domain((-1.0, -0.5, 0.0), upper, n, N, mg_levels=1, overlap=1)
        out = d.apply_f32(torch.from_numpy(u.ravel()).cuda()).cpu().numpy().astype(np.float64)
        err = np.linalg.norm(out - ref.ravel()) / np.linalg.norm(ref) / 2.0**-23
        assert err < 0.6, (n, err)
