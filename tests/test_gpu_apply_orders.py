"""The operator's passes that test_gpu_apply_ragged does not reach: second order on ragged 3-D grids, where the folded pass
stages planes of another size and depth by plain copies or the general pass runs, on both sides of the line between them in either
precision, and the walk by one warp over more than 2^18 rows of the walls' classes (both orders).  A stencil of order Q is exact
for polynomials of degree Q; bounds as there."""
import math

import numpy as np
import pytest

from test_gpu_apply_ragged import A, _avg, _full

pytestmark = pytest.mark.gpu


def _problem(n, order, inside):
    import paper_1411_4283_gb300 as P
    G = P.eb_geometry_spheres(n, [(0.503, 0.497, 0.501)], [0.44 if inside else 0.28], inside=inside, moment_degree=4)
    x = (np.arange(n) + 0.5) - 0.5 * n
    s = (x[None, None, :] * A[0] + x[None, :, None] * A[1] + x[:, None, None] * A[2]).reshape(-1)
    flag, cut, vol = G.table("flag"), G.table("cut_cells"), G.table("vol_mom")

    def avg(p):
        one = [np.dot(_full(3)[0], c) for c in _poly(p)]  # the average about s is a polynomial of s
        out = sum(c * s ** (p - j) for j, c in enumerate(one))
        out[cut] = _avg(vol, range(3), s[cut], p)
        return out

    kappa = (flag == 1).astype(float)
    kappa[cut] = vol[:, 0]
    phi, lap = avg(order), order * (order - 1) * (A ** 2).sum() * n ** 2 * kappa * avg(order - 2)
    st = P.eb_build_stencils(G, order=order)
    ids, base, g_wall = P.eb_wall_faces(st), 0, []
    for d in range(3):
        m = [n + (k == d) for k in range(3)]
        f = ids[(ids >= base) & (ids < base + math.prod(m))] - base
        base += math.prod(m)
        sf = np.zeros(len(f))
        for k in range(3):
            i, f = f % m[k], f // m[k]
            sf += A[k] * (i - 0.5 * n + (0.0 if k == d else 0.5))
        g_wall.append(_avg(np.repeat(_full(2), len(sf), 0), [k for k in range(3) if k != d], sf, order))
    g_eb = _avg(G.table("eb_mom"), range(3), s[cut], order)
    return st, phi * (flag > 0), lap, g_eb, np.concatenate(g_wall), flag, kappa


def _poly(p):
    """Coefficients of (s + a . xi)^p by the power of a . xi, over the monomials of the tables."""
    from test_gpu_apply_ragged import _mons
    out = []
    for j in range(p + 1):
        c = np.zeros(len(_mons(3)))
        for i, m in enumerate(_mons(3)):
            if sum(m) == j:
                c[i] = math.comb(p, j) * math.factorial(j) / math.prod(math.factorial(v) for v in m) * math.prod(A ** np.array(m))
        out.append(c)
    return out


@pytest.mark.parametrize("n,order,inside", [(17, 2, False), (41, 2, True), (49, 2, False), (67, 2, False), (71, 2, True),
                                            (41, 4, True), (53, 4, True), (111, 4, False), (129, 2, False)])
def test_polynomial_is_exact(n, order, inside):
    import torch
    import paper_1411_4283_gb300 as P
    st, phi, lap, g_eb, g_wall, flag, kappa = _problem(n, order, inside)
    dev = lambda a, t=torch.float64: torch.as_tensor(a).to("cuda", t)  # noqa: E731
    bg = P.eb_bc_rhs(st, dev(g_eb), dev(g_wall if len(g_wall) else np.zeros(1)),
                     torch.empty(n ** 3, dtype=torch.float64, device="cuda"))
    x = dev(phi)
    y = P.eb_apply(st, x, torch.full_like(x, float("nan")), kappa_weighted=True)
    err = (y + bg).cpu().numpy() - lap
    assert np.all(np.isfinite(err))
    assert np.abs(err).max() <= 7e-11 * np.abs(phi).max() * n ** 2, np.abs(err).max() / n ** 2
    assert torch.all(y[dev(flag, torch.uint8) == 0] == 0)
    x = dev(np.random.default_rng(n).uniform(-1, 1, n ** 3) * (flag > 0))
    for kw in (True, False):
        y64 = P.eb_apply(st, x, torch.empty_like(x), kappa_weighted=kw)
        y32 = P.eb_apply(st, x.float(), torch.full_like(x.float(), float("nan")), kappa_weighted=kw)
        if not kw:
            y64, y32 = y64[dev(kappa) > 0.01], y32[dev(kappa) > 0.01]
        assert torch.linalg.norm(y32.double() - y64) <= 1e-5 * torch.linalg.norm(y64)
