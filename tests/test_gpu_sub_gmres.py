"""GPU parity of the subdomain GMRES (Sec. III.E, Laplacian approximation) against the oracle at the
iteration counts and column lengths its kernels distinguish."""
import pytest

from gpu_util import rand, rel
from oracle import dg, puncture, schwarz
from test_gpu_linearized import _dev, _setup

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,N,ov,m", [((3, 2, 2), 3, 1, 1), ((2, 2, 1), 4, 2, 2), ((2, 1, 2), 5, 2, 5), ((1, 1, 2), 8, 3, 3)])
def test_every_iteration_count_and_column_length_of_the_subdomain_gmres(n, N, ov, m):
    """One to five iterations (the last one combined in the scatter, three unrolled) and, at N = 8 with three
    layers in FP64, columns too long for registers; two linearizations on one domain, so that a diagonal kept
    from the first would show. Tolerances as above."""
    for precision, gemm, tol in (("fp64", "default", 1e-10), ("mixed", "simt", 1e-4)):
        d, grid, pr, u, _ = _setup(n, N, ov, 4.0, precision, gemm=gemm)
        lv = pr.schwarz[0]
        b, u0 = rand(65, (grid.n_elements, N, N, N)), rand(66, (grid.n_elements, N, N, N))
        d.set_subdomain_solver("gmres", m)
        for scale in (1.0, 3.0):
            D = pr.mass * puncture.source_deriv(scale * u, pr.alpha, pr.beta)
            lin = lambda x: dg.apply(pr.graphs[0], x) + D * x
            ref = lv.smooth(b, u0, 2, lin, schwarz.gmres_subdomain_solver(lv, D, m))
            d.set_linearization(_dev(scale * u))
            out = d.schwarz_smooth(0, _dev(b), _dev(u0), 2).cpu().numpy()
            assert rel(out, ref) < tol, (precision, scale)
