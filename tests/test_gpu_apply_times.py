"""The operator's time on small FP64 grids, each against a case of the same run that cannot differ much from it.  In 2-D the
passes of an apply take what one row's chain and one tile take until the grid fills the chip (29 us at 100^2 and at
300^2): applies that follow one another on 300^2 take at most 2.5 times those on 100^2 (1.0; with eight warps to a row
in FP64 it was 4.8, the SMs changing their shared memory's partition in turn).  On a small ragged 3-D grid inside
a sphere FP64 takes up to four times FP32 (2.2; the folded pass in pieces of eight planes took 6.9).  The boundary part on
4096^2 in second order, which zeroes a vector and writes some rows of it, takes at most 1.35 times a copy of the
vector (a warp for each short row: 1.6)."""
import pytest

pytestmark = pytest.mark.gpu


def _median(f):
    """Milliseconds of 40 calls one after the other, the median of nine times."""
    import torch
    ev = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
    out = []
    for _ in range(9):
        ev[0].record()
        for _ in range(40):
            f()
        ev[1].record()
        ev[1].synchronize()
        out.append(ev[0].elapsed_time(ev[1]))
    return sorted(out)[4]


def _time(dim, n, inside, dtype):
    import torch
    import paper_1411_4283_gb300 as P
    c = (0.503, 0.497, 0.501)[:dim]
    g = (P.eb_geometry_spheres if dim == 3 else P.eb_geometry_circles)(n, [c], [0.45 if inside else 0.3], inside=inside,
                                                                     moment_degree=4)
    st = P.eb_build_stencils(g, order=4)
    x = torch.rand(n ** dim, device="cuda", dtype=getattr(torch, dtype))
    y = torch.empty_like(x)
    return _median(lambda: P.eb_apply(st, x, y))


def test_boundary_part_in_2d():
    import torch
    import paper_1411_4283_gb300 as P
    n = 4096
    g = P.eb_geometry_circles(n, [(0.503, 0.497)], [0.3], moment_degree=4)
    st = P.eb_build_stencils(g, order=2)
    f64 = dict(dtype=torch.float64, device="cuda")
    ge, gw, y, x = torch.ones(g.n_cut, **f64), torch.ones(st.n_wall, **f64), torch.empty(n * n, **f64), torch.ones(n * n, **f64)
    assert _median(lambda: P.eb_bc_rhs(st, ge, gw, y)) <= 1.35 * _median(lambda: y.copy_(x))


def test_small_2d_grids_take_one_time():
    assert _time(2, 300, False, "float64") <= 2.5 * _time(2, 100, False, "float64")


def test_small_ragged_grid_in_fp64():
    assert _time(3, 29, True, "float64") <= 4.0 * _time(3, 29, True, "float32")
