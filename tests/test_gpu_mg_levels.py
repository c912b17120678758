"""The multigrid cycle at the sizes where its path changes: all levels inside one CTA or only the coarser ones
(4096 cells, and the shared memory that FP64 levels need), even and odd level sizes, and the first sweep and the
prolongation fused with the next sweep or passes of their own (FP64 above 65536 cells).  The FP32 and the FP64 cycle change the path of
a solve and not its answer: both solutions agree to 1e-9 of the largest value (the tolerance of the comparison of
preconditioners in test_gpu_parity), and the FP64 solve takes at most the 40 iterations allowed there."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim,n", [(2, 20), (2, 48), (2, 64), (2, 65), (2, 130), (2, 257), (3, 16), (3, 17), (3, 31), (3, 41)])
def test_cycle_changes_the_path_only(dim, n):
    import torch
    import paper_1411_4283_gb300 as P
    c = (0.513, 0.487, 0.505)[:dim]
    g = (P.eb_geometry_spheres if dim == 3 else P.eb_geometry_circles)(n, [c], [0.23], moment_degree=4)
    st = P.eb_build_stencils(g, order=4)
    gen = torch.Generator().manual_seed(n)
    rho = (torch.rand(n ** dim, generator=gen, dtype=torch.float64) - 0.5).cuda()
    rho *= torch.as_tensor(g.table("flag") > 0).cuda()
    ge = torch.zeros(g.n_cut, dtype=torch.float64, device="cuda")
    gw = torch.zeros(2 * dim * n ** (dim - 1), dtype=torch.float64, device="cuda")
    out = {}
    for mixed in (True, False):
        phi = torch.zeros(n ** dim, dtype=torch.float64, device="cuda")
        info = P.eb_solve(st, rho, ge, gw, phi, tol=1e-11, mixed=mixed)
        assert info["status"] == "EB_OK"
        out[mixed] = phi.cpu().numpy()
    assert np.abs(out[True] - out[False]).max() <= 1e-9 * np.abs(out[False]).max()
    assert info["iterations"] <= 40, info
