"""The least-squares stencils at any scale of the faces' moments.  Scaling the moments of the cut faces (normal
to the axes and EB) by a power of two scales the right-hand sides of their systems and nothing else (a row is
normalised by its own zeroth moment), and s = W (A^T W)^+ F is linear in F: the coefficients are the unscaled ones
times that power, to the last bit, because a power of two passes every rounding.  From 2^-40 on the scales are
below what squares of FP32 numbers hold, at 2^-200 and 2^140 below and above FP32 itself."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SHAPES = {
    # dim, n, order, path radius, Neumann: a warp per system and a block per system, few and many unknowns
    "warp_2d_q4": (2, 40, 4, 0, False),
    "block_2d_q2": (2, 40, 2, 3, False),
    "warp_3d_q2": (3, 17, 2, 0, False),
    "block_3d_q4": (3, 16, 4, 0, False),
}


def _tables(dim, n, inside=False):
    import paper_1411_4283_gb300 as P
    c = (0.51, 0.49, 0.503)[:dim]
    g = (P.eb_geometry_spheres if dim == 3 else P.eb_geometry_circles)(n, [c], [0.3], inside=inside, moment_degree=4)
    t = {k: g.table(k) for k in ("flag", "cut_cells", "vol_mom", "eb_mom", "eb_nmom")}
    t.update({k: [g.table(k, d) for d in range(dim)] for k in ("face_flag", "cut_faces", "face_mom")})
    return t


def _build(t, dim, n, scale, **kw):
    import paper_1411_4283_gb300 as P
    g = P.DeviceGeometry(dim, (n,) * dim, 1.0 / n, 4, t["flag"], t["cut_cells"], t["vol_mom"], t["eb_mom"],
                         t["eb_nmom"] * scale, t["face_flag"], t["cut_faces"], [f * scale for f in t["face_mom"]])
    return P.eb_build_stencils(g, **kw)


def _cut_faces(t, dim, n):
    base, out = 0, []
    for d in range(dim):
        f = np.asarray(t["cut_faces"][d], dtype=np.int64)
        out.append(base + f[:: max(1, len(f) // 20)])
        base += n ** (dim - 1) * (n + 1)
    out.append(base + np.arange(0, len(t["cut_cells"]), max(1, len(t["cut_cells"]) // 30)))
    return np.concatenate(out)


@pytest.mark.parametrize("name", list(SHAPES))
@pytest.mark.parametrize("e", [-40, -54, -66, -200, 70, 140])
def test_coefficients_scale_with_the_moments(name, e):
    import paper_1411_4283_gb300 as P
    dim, n, order, R, _ = SHAPES[name]
    t = _tables(dim, n)
    a = _build(t, dim, n, 1.0, order=order, path_radius=R)
    b = _build(t, dim, n, 2.0 ** e, order=order, path_radius=R)
    assert a.info["n_ls_fp64"] == b.info["n_ls_fp64"]  # the same systems were left to the FP64 kernel
    for f in _cut_faces(t, dim, n):
        ca, va = P.eb_stencil_query(a, int(f))
        cb, vb = P.eb_stencil_query(b, int(f))
        assert np.array_equal(ca, cb)
        assert np.array_equal(vb * 2.0 ** -e, va), (f, np.abs(vb * 2.0 ** -e - va).max() / np.abs(va).max())
