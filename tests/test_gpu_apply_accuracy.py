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


@pytest.mark.parametrize("upper", [(1.0, 1e-20, 1.0), (1.0, 1e20, 1.0), (1e-22, 1.0, 1e-21)])
def test_elements_too_thin_for_a_ratio_of_directions(upper):
    """Above 1 : 2^60 the directions keep their own factors: the operator is as right as elsewhere (1e-12, FP32 2e-5)."""
    n, N = (3, 2, 2), 5
    grid = dg.BoxGrid((0.0, 0.0, 0.0), upper, n, N, 1.5, (False,) * 6)
    u = rand(970, (grid.n_elements, N, N, N)).astype(np.float32).astype(np.float64)
    ref = dg.apply(grid.graph(), u).ravel()
    d = dgg.Domain((0.0, 0.0, 0.0), upper, n, N, mg_levels=1, overlap=1)
    t = torch.from_numpy(u.ravel()).cuda()
    for out, tol in ((d.apply(t), 1e-12), (d.apply_f32(t.float()).double(), 2e-5)):
        assert np.linalg.norm(out.cpu().numpy() / np.abs(ref).max() - ref / np.abs(ref).max()) <= tol * np.linalg.norm(
            ref / np.abs(ref).max())
