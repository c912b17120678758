"""Iterations of the refined solve (FP32 cycle) and of the FP64 solve where the multigrid cycle's path changes, the sizes of
test_gpu_mg_levels and two whose finest level is above 2^20 cells.  A cycle that smooths or transfers less well still converges, in
more iterations: the bounds are twice the counts of the cycle before its passes were fused and its coarse levels moved into shared
memory (the last digit of a sum moves a count by a few; 31^3 is left out, where weak cells make the refined solve take 55 to 130 from run
to run)."""
import pytest

pytestmark = pytest.mark.gpu

COUNTS = {  # (dimension, n): FP32 cycle, FP64 cycle
    (2, 20): (23, 15), (2, 48): (27, 18), (2, 64): (24, 17), (2, 65): (17, 19), (2, 130): (28, 18), (2, 257): (34, 22),
    (2, 1030): (48, 22), (3, 16): (20, 15), (3, 17): (21, 15), (3, 41): (24, 18), (3, 103): (29, 20)}


@pytest.mark.parametrize("dim,n", list(COUNTS))
def test_iterations(dim, n):
    import torch
    import paper_1411_4283_gb300 as P
    c = (0.513, 0.487, 0.505)[:dim]
    g = (P.eb_geometry_spheres if dim == 3 else P.eb_geometry_circles)(n, [c], [0.23], moment_degree=4)
    st = P.eb_build_stencils(g, order=4)
    rho = (torch.rand(n ** dim, generator=torch.Generator().manual_seed(n), dtype=torch.float64) - 0.5).cuda()
    rho *= torch.as_tensor(g.table("flag") > 0).cuda()
    f64 = dict(dtype=torch.float64, device="cuda")
    ge, gw = torch.zeros(g.n_cut, **f64), torch.zeros(st.n_wall, **f64)
    for mixed, count in zip((True, False), COUNTS[dim, n]):
        info = P.eb_solve(st, rho, ge, gw, torch.zeros_like(rho), tol=1e-11, mixed=mixed)
        assert info["iterations"] <= 2 * count, (mixed, info["iterations"])
