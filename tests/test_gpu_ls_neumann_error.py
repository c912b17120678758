"""The default least squares against the FP64 kernel on Neumann systems, whose terms cancel most: with the same rows, the two
operators on a rough field differ by the roundings of the solves.  The bounds are what the kernel before k_lsq_mixed (FP32 Householder
factor, FP64 corrections) had; two interleaved chains for a row's sum, and corrections of up to 5e-4 in pairs of FP32, exceeded them by 10 to
26 %."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim,n,inside,bound", [(3, 24, True, 4.17e-16), (3, 31, True, 4.18e-16), (3, 40, True, 5.18e-16),
                                                (2, 333, False, 9.26e-16)])
def test_operator_difference(dim, n, inside, bound):
    import torch
    import paper_1411_4283_gb300 as P
    make = P.eb_geometry_spheres if dim == 3 else P.eb_geometry_circles
    g = make(n, [(0.503, 0.497, 0.501)[:dim]], [0.45 if inside else 0.3], inside=inside, moment_degree=4)
    g.set_eb_bc(np.ones(g.n_cut, dtype=np.uint8))
    gen = torch.Generator("cuda").manual_seed(5)
    phi = torch.rand(n ** dim, generator=gen, device="cuda", dtype=torch.float64) * 2 - 1
    a, b = [P.eb_apply(P.eb_build_stencils(g, order=4, ls_precision=ls), phi, torch.empty_like(phi)) for ls in ("mixed", "fp64")]
    assert torch.linalg.norm(a - b) <= bound * torch.linalg.norm(b), (torch.linalg.norm(a - b) / torch.linalg.norm(b)).item()
