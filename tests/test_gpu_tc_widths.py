"""The tensor-core subdomain product at every tile width: classes of 16, 17, 32, 33, 48, 49, 64, 68, 128,
132, 192 and 196 subdomains (tiles of 16 to 128 columns, one or several equal parts of a class) against
the FP32 CUDA-core product, to the accuracy of TF32 inputs."""
import pytest
import torch

from gpu_util import box, rand, rel

pytestmark = pytest.mark.gpu

dgg = pytest.importorskip("paper_2111_06767_gb300")


@pytest.mark.parametrize("nx", [18, 19, 34, 35, 50, 51])
def test_class_sizes_at_the_tile_widths_match_simt(monkeypatch, nx):
    # nx - 2 subdomains touch no face of the box, 4 (nx - 2) one of its four long faces or edges each
    n, N = (nx, 3, 3), 4
    n_dof = box(n, N).n_elements * N**3
    b, u0 = (torch.from_numpy(rand(s, (n_dof,))).cuda() for s in (87, 88))
    ref = dgg.Domain(n=n, N=N, mg_levels=1, overlap=2, precision="mixed", gemm="simt")
    du_s = (ref.schwarz_smooth(0, b, u0.clone(), 1) - u0).cpu().numpy()
    for split in (1, 33):  # tiles of up to 64 and of up to 128 columns
        monkeypatch.setenv("DG_GEMM_SPLIT", str(split))
        d = dgg.Domain(n=n, N=N, mg_levels=1, overlap=2, precision="mixed", gemm="tf32")
        du_t = (d.schwarz_smooth(0, b, u0.clone(), 1) - u0).cpu().numpy()
        assert rel(du_t, du_s) < 3e-3, split
