"""The library's performance cases: what its users have it do, through the package's public entry points.

Kinds of a case (the moment tables come from the library's device generators, as a user's would):
  apply     the operator on a vector, in the Krylov dtype (FP32) or the refinement's (FP64);
  residual  the FP64 operator and the boundary part B g, as a truncation study evaluates them;
  build     all flux stencils and the operator of new moment tables, then one evaluation with it;
  solve     a Poisson solve on stencils in hand, from a zero guess;
  batch     many small 2-D geometries: one batched build, the batched solver's set-up and solve;
  geometry  the moment tables of new spheres, read back.
Geometries are the framework's own examples: the unit square minus one circle (r = 0.3 near its middle)
or five, the unit cube minus a sphere of radius 0.35, the inside of a sphere of radius 0.45.
"""
import math
import random

import numpy as np
import torch

import paper_1411_4283_gb300 as P


def listed():
    return [
        # the smallest calls: config-sized 2-D study, launches and latency only
        {"name": "residual2d_f64_32", "kind": "residual", "dim": 2, "n": 32, "order": 4, "bodies": "circle"},
        # a user's own Krylov method on an ordinary, ragged 3-D grid
        {"name": "apply3d_f32_100", "kind": "apply", "dim": 3, "n": 100, "order": 4, "bodies": "sphere", "dtype": "f32"},
        # the same on the benchmark's grid, the largest one
        {"name": "apply3d_f32_256", "kind": "apply", "dim": 3, "n": 256, "order": 4, "bodies": "sphere", "dtype": "f32"},
        # the FP64 operator that residuals and error studies need
        {"name": "apply3d_f64_160", "kind": "apply", "dim": 3, "n": 160, "order": 4, "bodies": "sphere", "dtype": "f64"},
        # stencils of the smallest 2-D study: one of many geometries in a loop
        {"name": "build2d_q4_32", "kind": "build", "dim": 2, "n": 32, "order": 4, "bodies": "circle"},
        # the finest grid of the second-order convergence sweep
        {"name": "build2d_q2_1024", "kind": "build", "dim": 2, "n": 1024, "order": 2, "bodies": "five"},
        # a moderate fourth-order 3-D build on an odd grid
        {"name": "build3d_q4_63", "kind": "build", "dim": 3, "n": 63, "order": 4, "bodies": "sphere"},
        # a large fourth-order 3-D build
        {"name": "build3d_q4_160", "kind": "build", "dim": 3, "n": 160, "order": 4, "bodies": "sphere"},
        # second order with Neumann data on the boundary, inside a sphere
        {"name": "build3d_q2_neumann_80", "kind": "build", "dim": 3, "n": 80, "order": 2, "bodies": "inside",
         "neumann": True},
        # time to solution of a 3-D problem, mixed precision
        {"name": "solve3d_mixed_128", "kind": "solve", "dim": 3, "n": 128, "order": 4, "bodies": "sphere",
         "mixed": True},
        # a parameter study: many 2-D geometries at once
        {"name": "batch2d_16", "kind": "batch", "dim": 2, "n": 160, "order": 4, "bodies": "circle", "count": 16},
        # the tables of a new 3-D geometry
        {"name": "geometry3d_96", "kind": "geometry", "dim": 3, "n": 96, "order": 4, "bodies": "sphere"},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["apply", "apply", "residual", "build", "build", "build", "solve", "batch", "geometry"])
    dim = 2 if kind == "batch" else 3 if kind == "geometry" else rng.choice([2, 3, 3])
    order = rng.choice([4, 4, 2]) if kind in ("apply", "residual", "build") else 4
    c = {"kind": kind, "dim": dim, "order": order}
    if dim == 3:
        low = 32 if kind == "geometry" else 24
        top = {"apply": 220, "residual": 150, "build": 150, "solve": 120, "geometry": 96}[kind]
        c["n"] = _log_int(rng, low, top)
        c["bodies"] = rng.choice(["sphere", "sphere", "inside"])
    elif kind == "batch":
        c["n"] = _log_int(rng, 48, 160)
        c["bodies"] = "circle"
        c["count"] = rng.randint(3, 16)
    else:
        c["n"] = _log_int(rng, 32, 320 if kind == "solve" else 1024)
        c["bodies"] = rng.choice(["circle", "five"]) if c["n"] >= 128 else "circle"
    if kind == "apply":
        c["dtype"] = rng.choice(["f32", "f32", "f64"])
    if kind == "solve":
        c["mixed"] = rng.random() < 0.7
    if kind == "build" and rng.random() < 0.25:
        c["neumann"] = True
    return c


def _bodies(case, rng, n):
    """(centres, radii, inside) of a seeded geometry on an n^dim grid."""
    h = 1.0 / n
    which = case["bodies"]
    if which == "sphere":
        return [tuple(0.5 + rng.uniform(-0.5 * h, 0.5 * h) for _ in range(3))], [0.35], False
    if which == "inside":
        return [tuple(0.5 + rng.uniform(-0.5 * h, 0.5 * h) for _ in range(3))], [0.45], True
    if which == "circle":
        return [(0.5 + rng.uniform(-0.05, 0.05), 0.5 + rng.uniform(-0.05, 0.05))], [rng.uniform(0.25, 0.3)], False
    cen, rad = [(0.51 + rng.uniform(-h, h), 0.49 + rng.uniform(-h, h))], [0.3]
    while len(rad) < 5:
        r, x, y = rng.uniform(0.05, 0.15), rng.random(), rng.random()
        if min(x, y) - r < 0.04 or max(x, y) + r > 0.96:
            continue
        if all(math.hypot(x - a, y - b) - r - s >= 0.04 for (a, b), s in zip(cen, rad)):
            cen.append((x, y))
            rad.append(r)
    return cen, rad, False


def _geometry(case, rng, n):
    cen, rad, inside = _bodies(case, rng, n)
    make = P.eb_geometry_spheres if case["dim"] == 3 else P.eb_geometry_circles
    g = make(n, cen, rad, inside=inside, moment_degree=4)
    if case.get("neumann"):
        g.set_eb_bc(np.ones(g.n_cut, dtype=np.uint8))
    return g


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _field(n, gen, dtype=torch.float64):
    return torch.rand(n, generator=gen, device="cuda", dtype=dtype) * 2 - 1


def _smooth(n, dim, gen):
    """Cell values of a smooth source: a product of sines with seeded phases."""
    x = (torch.arange(n, device="cuda", dtype=torch.float64) + 0.5) / n
    ph = torch.rand(3, generator=gen, device="cuda", dtype=torch.float64)
    s = [torch.sin(2 * math.pi * (x - ph[d])) for d in range(3)]
    f = s[1][:, None] * s[0][None, :]
    return (f if dim == 2 else s[2][:, None, None] * f[None]).reshape(-1).contiguous() * (-4 * math.pi ** 2 * dim)


def prepare(case, seed):
    rng, gen = random.Random(int(seed)), _gen(seed)
    kind, n, dim, order = case["kind"], case["n"], case["dim"], case["order"]
    if kind == "geometry":
        # mirrored and shifted by whole cells from seed to seed, which keeps the number of cut cells
        off = [rng.choice((-1, 1)) * v + rng.choice((-1, 0, 1)) for v in (0.137, 0.291, 0.383)]
        _, rad, inside = _bodies(case, rng, n)
        cen = [tuple(0.5 + v / n for v in off)]
        return {"case": case, "centers": cen, "radii": rad, "inside": inside}
    if kind == "batch":
        sizes = [max(32, int(round(n * 0.2 ** (k / max(1, case["count"] - 1))))) for k in range(case["count"])]
        geoms = [_geometry(case, rng, m) for m in sizes]
        return {"case": case, "geoms": geoms, "rho": [_smooth(m, 2, gen) for m in sizes],
                "g_eb": [_field(g.n_cut, gen) * 0.1 for g in geoms],
                "g_wall": [torch.zeros(4 * m, device="cuda", dtype=torch.float64) for m in sizes]}
    g = _geometry(case, rng, n)
    ncell = n ** dim
    s = {"case": case, "geom": g, "g_eb": _field(max(g.n_cut, 1), gen)}
    if kind != "build":
        s["st"] = P.eb_build_stencils(g, order=order)
    # the open wall faces: the whole box's, or none inside a body
    s["g_wall"] = _field(1 if case["bodies"] == "inside" else 2 * dim * n ** (dim - 1), gen)
    if kind == "solve":
        s["rho"] = _smooth(n, dim, gen)
        s["g_eb"] *= 0.1
        s["g_wall"].zero_()
    else:
        s["phi"] = _field(ncell, gen, torch.float32 if case.get("dtype") == "f32" else torch.float64)
    return s


def run(s):
    case = s["case"]
    kind = case["kind"]
    f64 = dict(dtype=torch.float64, device="cuda")
    if kind == "apply":
        return P.eb_apply(s["st"], s["phi"], torch.empty_like(s["phi"]), kappa_weighted=True)
    if kind == "residual":
        y = P.eb_apply(s["st"], s["phi"], torch.empty_like(s["phi"]), kappa_weighted=False)
        return [y, P.eb_bc_rhs(s["st"], s["g_eb"], s["g_wall"], torch.empty_like(y), kappa_weighted=False)]
    if kind == "build":
        st = P.eb_build_stencils(s["geom"], order=case["order"])
        y = P.eb_apply(st, s["phi"], torch.empty_like(s["phi"]), kappa_weighted=True)
        return [y, P.eb_bc_rhs(st, s["g_eb"], s["g_wall"], torch.empty_like(y), kappa_weighted=True)]
    if kind == "solve":
        phi = torch.zeros(s["rho"].numel(), **f64)
        P.eb_solve(s["st"], s["rho"], s["g_eb"], s["g_wall"], phi, tol=1e-11, mixed=case["mixed"])
        return phi
    if kind == "batch":
        sts = P.eb_build_stencils_batch(s["geoms"], order=case["order"])
        phis = [torch.zeros_like(r) for r in s["rho"]]
        P.BatchSolver(sts).solve(s["rho"], s["g_eb"], s["g_wall"], phis, tol=1e-11)
        return phis
    g = P.eb_geometry_spheres(case["n"], s["centers"], s["radii"], inside=s["inside"], moment_degree=4)
    out = {k: g.table(k) for k in ("flag", "cut_cells", "vol_mom", "eb_mom", "eb_nmom")}
    for d in range(3):
        for k in ("face_flag", "cut_faces", "face_mom"):
            out[f"{k}{d}"] = g.table(k, d)
    return out


def _sizes(case):
    """(cells with fluid, cut cells, rows of their own, least-squares systems, rows of one, K, footprint)."""
    n, dim, order = case["n"], case["dim"], case["order"]
    area, fluid = {"sphere": (1.539, 0.820), "inside": (2.545, 0.382), "circle": (1.73, 0.76),
                   "five": (4.4, 0.58)}[case["bodies"]]
    surf, R = area * n ** (dim - 1), 3 if order == 4 else 2
    K = {(2, 2): 6, (4, 2): 15, (2, 3): 10, (4, 3): 35}[(order, dim)]
    rows = 1.05 * (2 * R + 2) * (2 * R + 1) ** (dim - 1)
    own = min(fluid * n ** dim, surf * (2 * R + 1.3))
    foot = {(2, 2): 45, (4, 2): 77, (2, 3): 275, (4, 3): 637}[(order, dim)]
    return fluid * n ** dim, 1.5 * surf, own, (dim - 0.2) * own, rows, K, foot


def work(case):
    n, dim = case["n"], case["dim"]
    if case["kind"] == "batch":
        m = case["count"]
        one = [work({**case, "kind": "build", "n": max(32, int(round(n * 0.2 ** (k / max(1, m - 1)))))}) for k in range(m)]
        return {"bytes": sum(w["bytes"] for w in one), "flops": sum(w["flops"] for w in one)}
    cells, cut, own, systems, rows, K, foot = _sizes(case)
    tables = n ** dim * (1 + dim) + cut * (8 * K * (2 + dim) + 8 * 15 * dim)
    size = 4 if case.get("dtype") == "f32" else 8
    once = {"bytes": 2 * n ** dim * size + own * foot * size, "flops": 2 * foot * cells}
    if case["kind"] in ("apply", "residual"):
        return once
    if case["kind"] == "build":  # one QR, triangular solve and application of Q per system
        return {"bytes": tables + once["bytes"], "flops": once["flops"] + systems * (2 * rows * K * K + 4 * rows * K)}
    if case["kind"] == "solve":  # tens of operator applications, about as many again for the preconditioner
        return {"bytes": 30 * (2 * n ** dim * 4 + own * foot * 4), "flops": 30 * once["flops"]}
    return {"bytes": tables, "flops": cut * 48 * 48 * 3 * K * (2 + dim)}  # an area rule per patch


# ------------------------------------------------------------------ the method in 64 bits, plain torch
# Flux stencils s_f = W (A^T W)^+ F of every face and the flux divergence of a field with them, from the
# moment tables (the inputs), by a column-scaled QR (Cholesky, twice) of W A per system.


def _monomials(dim, q):
    out = []
    for deg in range(q + 1):
        def rec(prefix, left):
            if len(prefix) == dim - 1:
                out.append(prefix + (left,))
                return
            for p in range(left, -1, -1):
                rec(prefix + (p,), left - p)
        rec((), deg)
    return out


def _shift(mons, delta):
    """S with (moments of (x + delta)^p) = S (moments of x^q)."""
    S = np.zeros((len(mons), len(mons)))
    for i, p in enumerate(mons):
        for j, q in enumerate(mons):
            if all(a >= b for a, b in zip(p, q)):
                S[i, j] = math.prod(math.comb(a, b) * dl ** (a - b) for a, b, dl in zip(p, q, delta))
    return S


def _full(m):
    return math.prod(0.0 if q % 2 else 0.5 ** q / (q + 1) for q in m)


class _Method:
    def __init__(self, g, case):
        t = lambda a, dt: torch.as_tensor(np.ascontiguousarray(a)).to("cuda", dt)  # noqa: E731
        D = self.D = case["dim"]
        n = self.n = case["n"]
        self.shape = (n if D == 3 else 1, n, n)
        self.h = 1.0 / n
        self.R = 3 if case["order"] == 4 else 2
        self.neumann = bool(case.get("neumann"))
        self.mons = _monomials(D, case["order"])
        self.K = K = len(self.mons)
        pos = {m: i for i, m in enumerate(self.mons)}
        self.flag = t(g.table("flag"), torch.long).reshape(self.shape)
        cut = t(g.table("cut_cells"), torch.long)
        self.cut = torch.full((n ** D,), -1, dtype=torch.long, device="cuda")
        self.cut[cut] = torch.arange(len(cut), device="cuda")
        self.cut_cells = cut
        self.vol = t(g.table("vol_mom"), torch.float64)[:, :K].contiguous()
        self.eb = t(g.table("eb_mom"), torch.float64)[:, :K].contiguous()
        self.ebn = t(g.table("eb_nmom"), torch.float64)[:, :, :K].contiguous()
        # rows and fluxes of degree-lowered monomials: grad xi^p = p_d xi^(p - e_d)
        self.lower = torch.zeros(D, K, K, dtype=torch.float64, device="cuda")
        for i, m in enumerate(self.mons):
            for d in range(D):
                if m[d]:
                    self.lower[d, i, pos[tuple(v - (k == d) for k, v in enumerate(m))]] = m[d]
        # per direction: face flags, areas' tangential moments as D-dimensional moments about the face centre
        self.ff, self.fmom, self.fcut, self.fbase = [], [], [], [0]
        tmons = _monomials(D - 1, 4)
        for d in range(D):
            shp = tuple(s + (2 - ax == d) for ax, s in enumerate(self.shape))
            self.ff.append(t(g.table("face_flag", d), torch.long).reshape(shp))
            cf = t(g.table("cut_faces", d), torch.long)
            fm = t(g.table("face_mom", d), torch.float64).reshape(len(cf), -1)
            sel = [tmons.index(tuple(v for k, v in enumerate(m) if k != d)) if m[d] == 0 else -1 for m in self.mons]
            tab = torch.zeros(len(cf) + 1, K, dtype=torch.float64, device="cuda")
            for i, s in enumerate(sel):
                if s >= 0:
                    tab[:-1, i] = fm[:, s]
                    tab[-1, i] = _full(tmons[s])
            self.fmom.append(tab)  # last: the full face
            of = torch.full((math.prod(shp),), len(cf), dtype=torch.long, device="cuda")
            of[cf] = torch.arange(len(cf), device="cuda")
            self.fcut.append(of)
            self.fbase.append(self.fbase[-1] + math.prod(shp))
        self.full_vol = torch.tensor([_full(m) for m in self.mons], dtype=torch.float64, device="cuda")
        self._S = {}

    def S(self, delta):
        if delta not in self._S:
            self._S[delta] = torch.tensor(_shift(self.mons, delta), device="cuda")
        return self._S[delta]

    def face_index(self, d, x):
        """Local index of the face normal to d at coordinates x = (x, y, z)."""
        m0, m1 = self.n + (d == 0), self.n + (d == 1)
        return x[0] + m0 * (x[1] + m1 * x[2])

    def cell_index(self, x):
        return x[0] + self.n * (x[1] + self.n * x[2])

    def reach(self, x, ok):
        """[c, S, S, S] (z, y, x): cells of the box around x reached through open faces inside it."""
        R, D = self.R, self.D
        o = torch.arange(-R, R + 1, device="cuda")
        oz = o if D == 3 else o[R:R + 1]
        n = self.n
        cx = x[0][:, None, None, None] + o[None, None, None, :]
        cy = x[1][:, None, None, None] + o[None, None, :, None]
        cz = x[2][:, None, None, None] + oz[None, :, None, None]
        nz = self.shape[0]
        inside = (cx >= 0) & (cx < n) & (cy >= 0) & (cy < n) & (cz >= 0) & (cz < nz)
        ix, iy, iz = cx.clamp(0, n - 1), cy.clamp(0, n - 1), cz.clamp(0, nz - 1)
        vol = inside & (self.flag[iz, iy, ix] > 0)
        opens = []
        for d in range(D):
            c = [ix, iy, iz]
            c[d] = c[d] + 1
            opens.append(inside & (self.ff[d][c[2], c[1], c[0]] > 0))
        m = torch.zeros_like(vol)
        zc = R if D == 3 else 0
        m[:, zc, R, R] = ok & vol[:, zc, R, R]
        while True:
            new = m.clone()
            for d in range(D):
                ax = 3 - d
                lo, hi = [slice(None)] * 4, [slice(None)] * 4
                lo[ax], hi[ax] = slice(None, -1), slice(1, None)
                lo, hi = tuple(lo), tuple(hi)
                new[hi] |= m[lo] & opens[d][lo] & vol[hi]
                new[lo] |= m[hi] & opens[d][lo] & vol[lo]
            if bool((new == m).all()):
                return m
            m = new

    def stencils(self, d, x):
        """Stencils of the faces normal to d at x (d = None: EB faces of the cells x), padded rows:
        (coefficients, kinds, offsets) with kind 0 volume, 1 EB, 2 + 2 wd + side wall."""
        D, R, K, n = self.D, self.R, self.K, self.n
        c = len(x[0])
        dev = "cuda"
        if d is None:
            mask = self.reach(x, torch.ones(c, dtype=torch.bool, device=dev))
            low = [-R, -R, -R if D == 3 else 0]
            x0 = (0.0, 0.0, 0.0)
        else:
            xl = list(x)
            xl[d] = x[d] - 1
            hi = self.reach([v.clamp(0, s - 1) for v, s in zip(x, (n, n, self.shape[0]))], x[d] < n)
            lo = self.reach([v.clamp(0, s - 1) for v, s in zip(xl, (n, n, self.shape[0]))], xl[d] >= 0)
            ax = 3 - d
            pad = list(hi.shape)
            pad[ax] = 1
            z = torch.zeros(pad, dtype=torch.bool, device=dev)
            mask = torch.cat([z, hi], ax) | torch.cat([lo, z], ax)
            low = [-R, -R, -R if D == 3 else 0]
            low[d] -= 1
            x0 = tuple(-0.5 if k == d else 0.0 for k in range(3))
        sh = mask.shape[1:]
        sysm, flat = mask.reshape(c, -1).nonzero(as_tuple=True)
        off = [flat % sh[2] + low[0], flat // sh[2] % sh[1] + low[1], flat // (sh[1] * sh[2]) + low[2]]
        cell = [x[k][sysm] + off[k] for k in range(3)]
        cid = self.cell_index(cell)
        kinds = [torch.zeros_like(sysm)]
        where = [torch.arange(len(sysm), device=dev)]
        cu = self.cut[cid]
        w = (cu >= 0).nonzero()[:, 0]
        kinds.append(torch.ones_like(w))
        where.append(w)
        for wd in range(D):
            for side in range(2):
                at = (cell[wd] == (n - 1 if side else 0)).nonzero()[:, 0]
                f = [v[at] for v in cell]
                f[wd] = f[wd] + side
                at = at[self.ff[wd][f[2], f[1], f[0]] > 0]
                kinds.append(torch.full_like(at, 2 + 2 * wd + side))
                where.append(at)
        kind, where = torch.cat(kinds), torch.cat(where)
        sysm, off, cid, cell = sysm[where], [o[where] for o in off], cid[where], [v[where] for v in cell]
        rows = torch.zeros(len(kind), K, dtype=torch.float64, device=dev)
        wts = torch.zeros(len(kind), dtype=torch.float64, device=dev)
        code = kind + 16 * ((off[0] + 8) + 32 * ((off[1] + 8) + 32 * (off[2] + 8)))
        order = torch.argsort(code, stable=True)
        vals, counts = torch.unique_consecutive(code[order], return_counts=True)
        at = 0
        for v, k in zip(vals.tolist(), counts.tolist()):
            idx = order[at:at + k]
            at += k
            kd, rest = v % 16, v // 16
            dl = [float(rest % 32 - 8) - x0[0], float(rest // 32 % 32 - 8) - x0[1], float(rest // 1024 - 8) - x0[2]]
            if kd >= 2:
                dl[(kd - 2) // 2] += 0.5 if kd % 2 else -0.5
            r = math.sqrt(sum(q * q for q in dl[:D]))
            wt = 1.0 if r < 0.5 else (2.0 * r) ** -5
            St = self.S(tuple(dl[:D])).T
            if kd == 0:
                cq = self.cut[cid[idx]]
                mom = torch.where((cq >= 0)[:, None], self.vol[cq.clamp(min=0)] if len(self.vol) else 0.0, self.full_vol)
                m = mom @ St
                m = m / m[:, :1]
            elif kd == 1:
                cq = self.cut[cid[idx]]
                m0 = (self.eb[cq] @ St)
                if self.neumann:
                    m = sum((self.ebn[cq, e] @ St) @ self.lower[e].T for e in range(D)) / self.eb[cq, :1]
                    wt /= self.h
                else:
                    m = m0 / m0[:, :1]
            else:
                wd, side = (kd - 2) // 2, kd % 2
                f = [u[idx] for u in cell]
                f[wd] = f[wd] + side
                m = self.fmom[wd][self.fcut[wd][self.face_index(wd, f)]] @ St
                m = m / m[:, :1]
            rows[idx] = wt * m
            wts[idx] = wt
        # padded systems
        o2 = torch.argsort(sysm, stable=True)
        cnt = torch.bincount(sysm, minlength=c)
        start = torch.cumsum(cnt, 0) - cnt
        ss = sysm[o2]
        j = torch.arange(len(ss), device=dev) - start[ss]
        N = int(cnt.max())
        B = torch.zeros(c, N, K, dtype=torch.float64, device=dev)
        B[ss, j] = rows[o2]
        del rows
        W = torch.zeros(c, N, dtype=torch.float64, device=dev)
        W[ss, j] = wts[o2]
        kd = torch.full((c, N), -1, dtype=torch.long, device=dev)
        kd[ss, j] = kind[o2]
        of = torch.zeros(3, c, N, dtype=torch.long, device=dev)
        for q in range(3):
            of[q][ss, j] = off[q][o2]
        if d is None:
            cq = self.cut[self.cell_index(x)]
            F = sum(self.ebn[cq, e] @ self.lower[e].T for e in range(D))
        else:
            F = self.fmom[d][self.fcut[d][self.face_index(d, x)]] @ self.lower[d].T
        sc = B.norm(dim=1)
        B = B / sc[:, None, :]
        t = (F / sc)[:, :, None]
        for _ in range(2):  # B = Q R, twice: the second pass restores orthogonality
            L = torch.linalg.cholesky(B.transpose(1, 2) @ B)
            B = torch.linalg.solve_triangular(L, B.transpose(1, 2), upper=False).transpose(1, 2)
            t = torch.linalg.solve_triangular(L, t, upper=False)
        return W * (B @ t)[:, :, 0], kd, of

    def flux(self, s, kd, of, x, phi, g_eb, wall):
        """(stencil on the field, stencil on the boundary data) of faces at x with rows (s, kd, of)."""
        cell = [x[k][:, None] + of[k] for k in range(3)]
        n = self.n
        cid = self.cell_index([v.clamp(0, n - 1) for v in cell[:2]] + [cell[2].clamp(0, self.shape[0] - 1)])
        a = (s * torch.where(kd == 0, phi[cid], 0.0)).sum(1)
        cq = self.cut[cid]
        b = torch.where(kd == 1, g_eb[cq.clamp(min=0)] * (self.h if self.neumann else 1.0), 0.0)
        if bool((kd >= 2).any()):
            for wd in range(self.D):
                for side in range(2):
                    m = (kd == 2 + 2 * wd + side).nonzero(as_tuple=True)
                    f = [v[m] for v in cell]
                    f[wd] = f[wd] + side
                    b[m] = wall[self.fbase[wd] + self.face_index(wd, f)]
        return a, (s * b).sum(1)

    def evaluate(self, phi, g_eb, g_wall, weighted):
        """(L phi, B g), kappa-weighted or not."""
        D, n, R = self.D, self.n, self.R
        dev = "cuda"
        phi = phi.double()
        wall = torch.zeros(self.fbase[-1], dtype=torch.float64, device=dev)
        ids = []
        for d in range(D):
            for side in (0, n):
                m = torch.zeros_like(self.ff[d], dtype=torch.bool)
                m.select(2 - d, side).fill_(True)
                ids.append(self.fbase[d] + (m & (self.ff[d] > 0)).reshape(-1).nonzero()[:, 0])
        ids = torch.sort(torch.cat(ids))[0]
        wall[ids] = g_wall[:len(ids)]
        y = torch.zeros(2, n ** D, dtype=torch.float64, device=dev)
        far = (self.flag != 1).float()[None, None]
        near = torch.nn.functional.max_pool3d(far, (2 * R + 1 if D == 3 else 1, 2 * R + 1, 2 * R + 1), 1,
                                              (R if D == 3 else 0, R, R))[0, 0] > 0

        def coords(idx, d):
            m0, m1 = n + (d == 0), n + (d == 1)
            return [idx % m0, idx // m0 % m1, idx // (m0 * m1)]

        def add(d, x, fl):
            for k in range(2):
                f = fl[k]
                ok = x[d] < n
                y[k].index_add_(0, self.cell_index([v[ok] for v in x]), -f[ok])
                xl = list(x)
                xl[d] = x[d] - 1
                ok = xl[d] >= 0
                y[k].index_add_(0, self.cell_index([v[ok] for v in xl]), f[ok])

        step = 40000 if D == 2 or self.K <= 10 else 16000
        for d in range(D):
            x = coords((self.ff[d].reshape(-1) > 0).nonzero()[:, 0], d)
            xl = list(x)
            xl[d] = x[d] - 1
            at = lambda v: [v[k].clamp(0, self.shape[2 - k] - 1) for k in range(3)]  # noqa: E731
            hi, lo = at(x), at(xl)
            own = (near[hi[2], hi[1], hi[0]] & (x[d] < n)) | (near[lo[2], lo[1], lo[0]] & (xl[d] >= 0))
            for part in own.nonzero()[:, 0].split(step):
                xs = [v[part] for v in x]
                add(d, xs, self.flux(*self.stencils(d, xs), xs, phi, g_eb, wall))
            rest = (~own).nonzero()[:, 0]
            if not len(rest):
                continue
            xs = [v[rest] for v in x]
            key = torch.zeros_like(rest)
            for k in range(D):  # distances to both walls, as far as a stencil sees
                lo_, hi_ = xs[k], (n if k == d else n - 1) - xs[k]
                key = (key * 8 + lo_.clamp(max=R + 2)) * 8 + hi_.clamp(max=R + 2)
            _, inv = torch.unique(key, return_inverse=True)
            ncls = int(inv.max()) + 1
            rep = torch.full((ncls,), len(rest), dtype=torch.long, device=dev)
            rep.scatter_reduce_(0, inv, torch.arange(len(rest), device=dev), "amin")
            cls = self.stencils(d, [v[rep] for v in xs])
            for part in torch.arange(len(rest), device=dev).split(200000):
                xp, i = [v[part] for v in xs], inv[part]
                add(d, xp, self.flux(cls[0][i], cls[1][i], cls[2][:, i], xp, phi, g_eb, wall))
        if len(self.cut_cells):
            xa = coords(self.cut_cells, None)
            if self.neumann:
                y[1].index_add_(0, self.cut_cells, self.eb[:, 0] * g_eb[:len(self.cut_cells)] * self.h)
            else:
                for part in torch.arange(len(self.cut_cells), device=dev).split(step):
                    xs = [v[part] for v in xa]
                    fl = self.flux(*self.stencils(None, xs), xs, phi, g_eb, wall)
                    for k in range(2):
                        y[k].index_add_(0, self.cut_cells[part], fl[k])
        y *= n * n
        y[:, self.flag.reshape(-1) == 0] = 0.0
        if not weighted:
            y[:, self.cut_cells] /= self.vol[:, 0]
        return y[0], y[1]


def exact(case, seed):
    if case["kind"] not in ("apply", "residual", "build") or case["dim"] == 3 and case["n"] > 160:
        return None  # solves and tables have no short closed form; larger grids take too long
    s = prepare({**case, "kind": "build"}, seed)
    a, b = _Method(s["geom"], case).evaluate(s["phi"], s["g_eb"], s["g_wall"], case["kind"] != "residual")
    return a if case["kind"] == "apply" else [a, b]
