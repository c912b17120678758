"""The device sphere tables where their rules change: every moment degree, arcs from a whole circle inside
one cell (the longest pieces) to a sphere of many cells (the shortest, fewest points), and the poles.
Closed forms: the patches add up to 4 pi r^2, the volumes to the unit cube's rest.  A table entry is good to
about 1e-14 (rounding of some hundred terms of size one), a sum over n cells of size-one entries to n 1e-14,
so relative to the sum itself (n / 1.5 or more) the totals hold to 1e-13; 1e-12 is asked for."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

BODIES = {
    "one_cell": (8, (0.56, 0.57, 0.55), 0.04, False),
    "pole_cells": (9, (0.5, 0.5, 0.5), 0.3, False),
    "medium": (33, (0.51, 0.49, 0.503), 0.35, False),
    "inside": (21, (0.5, 0.5, 0.5), 0.45, True),
    "fine": (120, (0.5012, 0.4991, 0.5003), 0.35, False),
}


@pytest.mark.parametrize("name", list(BODIES))
def test_totals_and_degrees(name):
    import paper_1411_4283_gb300 as P
    N, c, r, inside = BODIES[name]
    G = P.eb_geometry_spheres(N, [c], [r], inside=inside, moment_degree=4)
    vol, eb, ebn = G.table("vol_mom"), G.table("eb_mom"), G.table("eb_nmom")
    assert abs(eb[:, 0].sum() / N ** 2 / (4 * np.pi * r * r) - 1) <= 1e-12
    ball = 4 / 3 * np.pi * r ** 3
    fluid = ((G.table("flag") == 1).sum() + vol[:, 0].sum()) / N ** 3
    assert abs(fluid - (ball if inside else 1 - ball)) <= 1e-12
    # lower degrees hold the same moments: two roundings of the same sums
    for q in range(4):
        H = P.eb_geometry_spheres(N, [c], [r], inside=inside, moment_degree=q)
        K, K2 = (q + 1) * (q + 2) * (q + 3) // 6, (q + 1) * (q + 2) // 2
        assert np.array_equal(H.table("cut_cells"), G.table("cut_cells"))
        assert np.abs(H.table("vol_mom") - vol[:, :K]).max() <= 1e-13
        assert np.abs(H.table("eb_mom") - eb[:, :K]).max() <= 1e-13
        assert np.abs(H.table("eb_nmom") - ebn[:, :, :K]).max() <= 1e-13
        for d in range(3):
            if G.desc.n_cutface[d] == 0:  # a sphere inside one cell cuts no face
                assert H.desc.n_cutface[d] == 0
                continue
            assert np.abs(H.table("face_mom", d) - G.table("face_mom", d)[:, :K2]).max() <= 1e-13
