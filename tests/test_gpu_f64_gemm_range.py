"""The FP64 subdomain product on the tensor cores at the ends of its operands' range, against the CUDA-core product."""
import numpy as np
import pytest
import torch

from gpu_util import rand

pytestmark = pytest.mark.gpu

dgg = pytest.importorskip("paper_2111_06767_gb300")


def test_an_inverse_that_is_not_finite_reaches_the_same_points():
    """Elements 1e155 times as long as wide: the subdomain matrices, built at unit width, overflow (their volume is
    1e310) and the inverses hold NaNs, while the operator itself stays finite. The NaNs have to reach the correction,
    not to vanish from it."""
    n, N = (5, 4, 4), 6
    b = torch.from_numpy(rand(920, (n[0] * n[1] * n[2] * N**3,))).cuda()
    finite = {}
    for gemm in ("simt", "default"):
        d = dgg.Domain((0.0, 0.0, 0.0), (5e-155, 4.0, 4.0), n, N, mg_levels=1, overlap=2, gemm=gemm)
        finite[gemm] = torch.isfinite(d.schwarz_smooth(0, b, torch.zeros_like(b), 1)).cpu().numpy()
    assert not finite["simt"].all()
    assert np.array_equal(finite["default"], finite["simt"])
