"""The mixed least-squares kernel in each of its shapes against the FP64 kernel: a warp per system and a block
of four warps per system for every number of unknowns (the rows of the largest system decide: wide path
radii take the small systems to the block shape), systems of more than 448 rows (the longer factor), Neumann
rows, the inside of a body, and a batch of geometries of different sizes.
Both solve the same systems to rounding times their condition: the coefficients agree to 1e-10 of a face's
largest, the bound the stencils are held to against the oracle."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

TOL = 1e-10
CASES = {
    # dim, n, order, path radius (0: the order's own), inside, Neumann; rows of the largest system from, to
    "warp_2d_q2": (2, 40, 2, 0, False, False, 30, 64),
    "warp_2d_q4": (2, 40, 4, 0, False, False, 65, 128),
    "warp_2d_q4_neumann": (2, 33, 4, 0, True, True, 40, 128),
    "block_2d_q2": (2, 40, 2, 3, False, False, 65, 640),
    "block_2d_q4": (2, 8, 4, 0, False, False, 129, 640),
    "warp_3d_q2": (3, 17, 2, 0, False, False, 100, 256),
    "warp_3d_q2_neumann": (3, 15, 2, 0, True, True, 100, 256),
    "block_3d_q2": (3, 15, 2, 3, True, False, 257, 640),
    "block_3d_q4": (3, 19, 4, 0, False, False, 449, 640),
    "block_3d_q4_neumann": (3, 16, 4, 0, True, True, 300, 640),
}


def _geometry(dim, n, inside, neumann, shift=0.0):
    import paper_1411_4283_gb300 as P
    if dim == 2 and n == 8:  # a circle on every second vertex cuts every cell, all of them in reach of the walls
        v = np.arange(1, 8, 2) / 8
        return P.eb_geometry_circles(8, [(x, y) for x in v for y in v], [0.05] * 16, moment_degree=4)
    c = (0.51 + shift, 0.49 - shift, 0.503)[:dim]
    make = P.eb_geometry_spheres if dim == 3 else P.eb_geometry_circles
    g = make(n, [c], [0.42 if inside else 0.3], inside=inside, moment_degree=4)
    if neumann:
        g.set_eb_bc(np.ones(g.n_cut, dtype=np.uint8))
    return g


def _agree(a, b, faces):
    import paper_1411_4283_gb300 as P
    for f in faces:
        ca, va = P.eb_stencil_query(a, int(f))
        cb, vb = P.eb_stencil_query(b, int(f))
        assert np.array_equal(ca, cb), f
        assert np.abs(va - vb).max() <= TOL * np.abs(vb).max(), (f, np.abs(va - vb).max() / np.abs(vb).max())


def _faces(g, n, dim):
    """EB faces and open grid faces, about 120 over the whole list."""
    base, out = 0, []
    for d in range(dim):
        f = np.nonzero(g.table("face_flag", d))[0]
        out.append(base + f[:: max(1, len(f) // 25)])
        base += n ** (dim - 1) * (n + 1)
    out.append(base + np.arange(0, g.n_cut, max(1, g.n_cut // 40)))
    return np.concatenate(out)


@pytest.mark.parametrize("name", list(CASES))
def test_mixed_equals_fp64(name):
    import paper_1411_4283_gb300 as P
    dim, n, order, R, inside, neumann, lo, hi = CASES[name]
    g = _geometry(dim, n, inside, neumann)
    a = P.eb_build_stencils(g, order=order, path_radius=R)
    b = P.eb_build_stencils(g, order=order, path_radius=R, ls_precision="fp64")
    assert lo <= a.info["max_rows"] <= hi
    assert a.info["n_ls_fp64"] < 0.05 * b.info["n_ls_fp64"]  # the mixed kernel solved them itself
    _agree(a, b, _faces(g, n, dim))


@pytest.mark.parametrize("dim,order", [(2, 4), (3, 2)])
def test_batch_equals_single(dim, order):
    import paper_1411_4283_gb300 as P
    ns = (36, 20, 28) if dim == 2 else (14, 18)
    gs = [_geometry(dim, n, False, False, 0.01 * i) for i, n in enumerate(ns)]
    for g, n, st in zip(gs, ns, P.eb_build_stencils_batch(gs, order=order)):
        _agree(st, P.eb_build_stencils(g, order=order, ls_precision="fp64"), _faces(g, n, dim))
