"""The operator on grids of every alignment: for a quartic phi the stencils are exact, so kappa L phi + B g is
kappa times the average of its Laplacian in every cell, cut ones included, with all averages from the moment
tables.  A stencil reproduces the flux of such a polynomial to 1e-11 of it, a cell sums seven of them over
h^2: |error| <= 7e-11 max|phi| n^2.  The sizes leave tiles, runs and slabs of the passes whole, ragged or
missing, rows of phi of 4, 8 and 16 bytes' alignment, and more than one tile of x."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

A = np.array([0.7, -0.4, 0.5])


def _mons(dim, q=4):
    out = []
    for deg in range(q + 1):
        if dim == 1:
            out.append((deg,))
        elif dim == 2:
            out += [(deg - j, j) for j in range(deg + 1)]
        else:
            out += [(deg - i, i - j, j) for i in range(deg + 1) for j in range(i + 1)]
    return out


def _avg(mom, dirs, s, p):
    """Averages of (s + a . xi)^p for local moments mom [n][K] over the directions dirs, offsets s [n]."""
    mons = _mons(len(dirs))
    tot = np.zeros(len(s))
    for j in range(p + 1):
        loc = np.zeros(len(s))
        for i, m in enumerate(mons):
            if sum(m) == j:
                c = math.factorial(j) / math.prod(math.factorial(v) for v in m)
                loc += c * math.prod(A[d] ** v for d, v in zip(dirs, m)) * mom[:, i]
        tot += math.comb(p, j) * s ** (p - j) * loc / mom[:, 0]
    return tot


def _full(dim):
    return np.array([[math.prod(0.0 if v % 2 else 0.5 ** v / (v + 1) for v in m) for m in _mons(dim)]])


def _problem(dim, n, inside):
    import paper_1411_4283_gb300 as P
    c = (0.503, 0.497, 0.501)[:dim]
    r = 0.44 if inside else 0.28
    G = (P.eb_geometry_spheres if dim == 3 else P.eb_geometry_circles)(n, [c], [r], inside=inside, moment_degree=4)
    x = (np.arange(n) + 0.5) - 0.5 * n  # cell centres in units of h
    s = x[None, :] * A[0] + x[:, None] * A[1] if dim == 2 else (x[None, None, :] * A[0] + x[None, :, None] * A[1]
                                                                + x[:, None, None] * A[2])
    s = s.reshape(-1)
    flag, cut = G.table("flag"), G.table("cut_cells")
    phi = _avg(np.repeat(_full(dim), n ** dim, 0), range(dim), s, 4)
    lap = _avg(np.repeat(_full(dim), n ** dim, 0), range(dim), s, 2)
    vol = G.table("vol_mom")
    phi[cut], lap[cut] = _avg(vol, range(dim), s[cut], 4), _avg(vol, range(dim), s[cut], 2)
    kappa = (flag == 1).astype(float)
    kappa[cut] = vol[:, 0]
    lap *= 12 * (A[:dim] ** 2).sum() * n ** 2 * kappa  # in units of h: the Laplacian's 1 / h^2
    g_eb = _avg(G.table("eb_mom"), range(dim), s[cut], 4)
    st = P.eb_build_stencils(G, order=4)
    ids, base, g_wall = P.eb_wall_faces(st), 0, []
    for d in range(dim):
        m = [n + (k == d) for k in range(dim)]
        f = ids[(ids >= base) & (ids < base + math.prod(m))] - base
        base += math.prod(m)
        sf = np.zeros(len(f))
        for k in range(dim):
            i, f = f % m[k], f // m[k]
            sf += A[k] * (i - 0.5 * n + (0.0 if k == d else 0.5))
        g_wall.append(_avg(np.repeat(_full(dim - 1), len(sf), 0), [k for k in range(dim) if k != d], sf, 4))
    st.kappa = kappa
    return st, phi * (flag > 0), lap, g_eb, np.concatenate(g_wall), flag


@pytest.mark.parametrize("dim,n,inside", [(3, 16, False), (3, 17, False), (3, 18, False), (3, 23, False), (3, 28, True),
                                          (3, 29, True), (3, 67, False), (3, 70, True), (3, 71, True), (3, 72, False), (3, 101, False),
                                          (2, 16, False), (2, 33, False), (2, 50, True), (2, 131, False)])
def test_quartic_is_exact(dim, n, inside):
    import torch
    import paper_1411_4283_gb300 as P
    st, phi, lap, g_eb, g_wall, flag = _problem(dim, n, inside)
    dev = lambda a, t=torch.float64: torch.as_tensor(a).to("cuda", t)  # noqa: E731
    big = np.abs(phi).max()
    bg = P.eb_bc_rhs(st, dev(g_eb), dev(g_wall if len(g_wall) else np.zeros(1)), torch.empty(n ** dim, dtype=torch.float64,
                                                                                               device="cuda"))
    x = dev(phi)
    y = P.eb_apply(st, x, torch.full_like(x, float("nan")), kappa_weighted=True)
    err = (y + bg).cpu().numpy() - lap
    assert np.all(np.isfinite(err))
    assert np.abs(err).max() <= 7e-11 * big * n ** 2, np.abs(err).max() / n ** 2
    assert torch.all(y[dev(flag, torch.uint8) == 0] == 0)
    # FP32 against FP64 on a rough field, both weightings, 1e-5 normwise (as against the oracle's operator)
    x = dev(np.random.default_rng(n).uniform(-1, 1, n ** dim) * (flag > 0))
    for kw in (True, False):
        y64 = P.eb_apply(st, x, torch.empty_like(x), kappa_weighted=kw)
        y32 = P.eb_apply(st, x.float(), torch.full_like(x.float(), float("nan")), kappa_weighted=kw)
        if not kw:  # without kappa the rows of tiny cells outweigh all others: compare the others
            big_cells = dev(st.kappa) > 0.01
            y64, y32 = y64[big_cells], y32[big_cells]
        assert torch.linalg.norm(y32.double() - y64) <= 1e-5 * torch.linalg.norm(y64)
