"""The FP64 subdomain product on the tensor cores at the ends of its operands' range, against the CUDA-core product."""
import math

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


def _step(n, N, ov, gemm, **box):
    """One smoothing step from u = 0 as a function of b."""
    d = dgg.Domain(n=n, N=N, mg_levels=1, overlap=ov, gemm=gemm, **box)
    return lambda b: d.schwarz_smooth(0, torch.from_numpy(b).cuda(), torch.zeros(d.n_dof, dtype=torch.float64).cuda(),
                                      1).cpu().numpy()


def _halves(x):
    hi = x * (2.0**27 + 1.0)
    hi = hi - (hi - x)
    return hi, x - hi


def _exact_rows(P, b):
    """P b, every row summed without rounding (products split into four exact ones)."""
    (Ph, Pl), (bh, bl) = _halves(P), _halves(b)
    return np.array([math.fsum(r) for r in np.concatenate([Ph * bh, Ph * bl, Pl * bh, Pl * bl], axis=1)])


def test_every_component_keeps_fp64_accuracy():
    """One step from u = 0 is a matrix P times b. At points that one subdomain covers, the CUDA-core product of a unit
    vector gives P_ik = w_i (s A^-1_ik), two roundings from exact, and P b is summed here without rounding. The digit
    product may round s A^-1_ik, its own result and its product with w_i: together 5, so 6 * 2^-53 (|P| |b|)_i
    bounds every component, whatever the range of b."""
    n, N, ov = (2, 1, 1), 6, 2
    m = n[0] * n[1] * n[2] * N**3
    x = np.arange(m) % N
    one = np.where(np.arange(m) < m // 2, x < N - ov, x >= ov)  # outside the other element's subdomain
    cuda_cores, digits = _step(n, N, ov, "simt"), _step(n, N, ov, "default")
    P = np.stack([cuda_cores(e) for e in np.eye(m)], axis=1)[one]
    points = np.eye(m)[[0, 7, m // 2 - 1, m // 2, m - 44]] * (2.0 / 3.0)
    rough = rand(921, (m,))
    decades = rough * 10.0 ** rand(922, (m,), -12.0, 0.0)
    tail = rough * np.exp(-np.linspace(0.0, 8.0, m) ** 2)
    for b in (*points, rough, decades, tail):
        err = np.abs(digits(b)[one] - _exact_rows(P, b))
        assert (err <= 6 * 2.0**-53 * (np.abs(P) @ np.abs(b))).all()


@pytest.mark.parametrize("n,N,ov,upper", [((3, 3, 2), 6, 5, (60.0, 3.0, 2.0)), ((20, 20, 20), 2, 1, (1.0, 1.0, 1.0))])
def test_levels_that_keep_the_cuda_core_product(monkeypatch, n, N, ov, upper):
    """Long thin elements with a wide overlap, where the entries of an inverse's row span more than 2^44, and N = 2 above
    one wave of tiles keep the CUDA-core product bit for bit (its K split pinned)."""
    monkeypatch.setenv("DG_GEMM_SPLIT", "1")
    b = rand(923, (n[0] * n[1] * n[2] * N**3,))
    out = [_step(n, N, ov, gemm, lower=(0.0, 0.0, 0.0), upper=upper)(b) for gemm in ("simt", "default")]
    assert np.array_equal(*out)
