"""FP64 subdomain product on the tensor cores (exact digit slices) against the CUDA-core product.

Two Schwarz steps on domains that differ only in `gemm`: class column counts around the tile widths
(1, 15-17, 47-49 and more), strides that are no multiple of the 64-wide K chunk, one to four drains of
512 terms, Neumann faces and unequal widths. Both products are FP64-accurate, so the steps agree to
1e-12 (the smoother's own tests allow 1e-10 against the oracle). The method is linear and powers of two
are exact, so scaled inputs give scaled outputs bit for bit; a NaN or an infinity reaches the same points.
"""
import numpy as np
import pytest
import torch

from gpu_util import rand, rel

pytestmark = pytest.mark.gpu

dgg = pytest.importorskip("paper_2111_06767_gb300")

CASES = [((1, 1, 3), 4, 1, ()), ((17, 3, 3), 4, 2, ()), ((8, 8, 8), 4, 1, (2,)), ((5, 4, 3), 5, 2, (0, 5)),
         ((9, 5, 5), 6, 2, ()), ((1, 1, 51), 7, 1, ()), ((2, 2, 2), 8, 2, ()), ((5, 5, 5), 8, 3, ()),
         ((3, 2, 3), 10, 4, (1,)), ((50, 1, 1), 3, 2, (4,))]


def _smooth(n, N, ov, neu, gemm, b, u):
    d = dgg.Domain((-1.0, -1.0, 0.0), (1.0, 1.5, 3.0), n, N, mg_levels=1, overlap=ov, neumann=neu, gemm=gemm)
    return d.schwarz_smooth(0, torch.from_numpy(b).cuda(), torch.from_numpy(u).cuda(), 2).cpu().numpy()


@pytest.mark.parametrize("n,N,ov,neu", CASES)
def test_tensor_core_product_matches_cuda_cores(n, N, ov, neu):
    m = n[0] * n[1] * n[2] * N**3
    b, u = rand(910, (m,)), rand(911, (m,))
    ref = _smooth(n, N, ov, neu, "simt", b, u)
    out = _smooth(n, N, ov, neu, "default", b, u)
    assert rel(out, ref) < 1e-12


def test_scaling_by_powers_of_two_is_exact_and_nonfinite_values_spread_alike():
    n, N = (5, 4, 4), 6
    m = n[0] * n[1] * n[2] * N**3
    b, u = rand(912, (m,)), rand(913, (m,))
    b[: m // 3] = 0.0
    out = _smooth(n, N, 2, (), "default", b, u)
    for k in (-300, 300):
        assert np.array_equal(_smooth(n, N, 2, (), "default", np.ldexp(b, k), np.ldexp(u, k)), np.ldexp(out, k))
    assert not _smooth(n, N, 2, (), "default", 0 * b, 0 * u).any()
    for bad in (np.nan, np.inf):
        c = b.copy()
        c[m // 2] = bad
        assert np.array_equal(np.isfinite(_smooth(n, N, 2, (), "default", c, u)),
                              np.isfinite(_smooth(n, N, 2, (), "simt", c, u)))
