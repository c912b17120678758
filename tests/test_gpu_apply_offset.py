"""The operator on vectors that start anywhere in a buffer: a field at an element's alignment but not at 16 bytes
gives what the same field at 16 bytes gives.  On grids whose rows have 16 bytes' length such a field does not suit
the tensor copies and vector loads of the aligned passes.  The passes sum a row in another order: 2 * 637 roundings of
2^-53 or 2^-24 of a row's terms at most, which the rough field and the rows' weights keep within 637 of the result's norm."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim,n,order", [(3, 16, 4), (3, 24, 2), (3, 70, 4), (2, 32, 4), (2, 64, 2)])
@pytest.mark.parametrize("dtype", ["float32", "float64"])
def test_field_at_an_odd_offset(dim, n, order, dtype):
    import torch
    import paper_1411_4283_gb300 as P
    c = (0.513, 0.487, 0.505)[:dim]
    g = (P.eb_geometry_spheres if dim == 3 else P.eb_geometry_circles)(n, [c], [0.28], moment_degree=4)
    st = P.eb_build_stencils(g, order=order)
    dt, ncell = getattr(torch, dtype), n ** dim
    x = (torch.rand(ncell, generator=torch.Generator().manual_seed(n), dtype=torch.float64) * 2 - 1).to("cuda", dt)
    eps = torch.finfo(dt).eps
    for kw in (True, False):
        want = P.eb_apply(st, x, torch.empty_like(x), kappa_weighted=kw)
        for off in (1, 2, 3):
            xs, ys = torch.zeros(ncell + 4, device="cuda", dtype=dt), torch.full((ncell + 4,), float("nan"), device="cuda", dtype=dt)
            xs[off:off + ncell] = x
            y = P.eb_apply(st, xs[off:off + ncell], ys[off:off + ncell], kappa_weighted=kw)
            assert torch.linalg.norm(y - want) <= 637 * eps * torch.linalg.norm(want)
            assert torch.isnan(ys[:off]).all() and torch.isnan(ys[off + ncell:]).all()


@pytest.mark.parametrize("mixed", [True, False])
def test_solution_at_an_odd_offset(mixed):
    import torch
    import paper_1411_4283_gb300 as P
    n = 24
    g = P.eb_geometry_spheres(n, [(0.513, 0.487, 0.505)], [0.28], moment_degree=4)
    st = P.eb_build_stencils(g, order=4)
    f64 = dict(dtype=torch.float64, device="cuda")
    rho, ge, gw = torch.ones(n ** 3, **f64), torch.zeros(g.n_cut, **f64), torch.zeros(st.n_wall, **f64)
    want, buf = torch.zeros(n ** 3, **f64), torch.zeros(n ** 3 + 1, **f64)
    P.eb_solve(st, rho, ge, gw, want, tol=1e-11, mixed=mixed)
    P.eb_solve(st, rho, ge, gw, buf[1:], tol=1e-11, mixed=mixed)
    assert (buf[1:] - want).abs().max() <= 1e-9 * want.abs().max()
