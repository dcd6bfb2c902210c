"""Coordinates, radii and spacings in other units than the angstrom, and patches
far larger than the spacing: the FP32 tests that leave pieces out have margins
that grow with the lengths they compare."""
import numpy as np
import pytest

import oracle
from paper_1809_04352_gb300 import build as libbuild
from paper_1809_04352_gb300 import eses, inputs

pytestmark = pytest.mark.gpu

TAU_TOL_A = 1e-6  # the root tolerance of every comparison with the oracle


@pytest.mark.parametrize("size", [1e3, 1e4, 3e4, 1e5])
@pytest.mark.parametrize("patch", [oracle.TYPE_F, oracle.TYPE_E, oracle.TYPE_V])
def test_patches_of_large_balls_in_fp64(patch, size):
    """A window of 29 x 27 x 25 points at spacing 1 around a point of a convex,
    a saddle and a concave patch of three balls of radius `size`."""
    libbuild.build()
    xyz = np.array([[-0.9, 0.0, 0.0], [0.9, 0.0, 0.0], [0.0, 1.3, 0.2]]) * size
    rad = np.array([1.0, 1.0, 0.8]) * size
    r_p = 0.7 * size
    start, way = {oracle.TYPE_F: ([0.0, 0.0, 0.0], [-1.0, -0.3, 0.4]), oracle.TYPE_E: ([0.0, 0.0, 0.0], [0.1, -1.0, 0.3]),
                  oracle.TYPE_V: ([0.0, 0.4, 0.0], [0.2, 0.3, 1.0])}[patch]
    start, way = np.array(start) * size, np.array(way) / np.linalg.norm(way)
    lo, hi = 0.0, 3.0 * size
    for _ in range(70):  # the surface on the ray
        mid = 0.5 * (lo + hi)
        if oracle.label_points(xyz, rad, r_p, (start + mid * way)[None])[0] == 1:
            lo = mid
        else:
            hi = mid
    origin = np.round(start + lo * way - [14.3, 12.2, 11.6]) + np.random.default_rng(3).random(3)
    dims = np.array([29, 27, 25])
    ref = oracle.run_on_grid(xyz, rad, r_p, 1.0, origin, dims)
    assert any((t == patch).any() for t in ref.ptype)
    ctx = eses.eses_create_on_grid(xyz, rad, r_p, 1.0, origin, dims)
    try:
        eses.eses_set_option(ctx, eses.ESES_OPT_PRECISION, eses.ESES_PREC_FP64)
        eses.eses_run(ctx)
        assert np.array_equal(eses.eses_labels(ctx), ref.labels)
        for a in range(3):
            g = eses.eses_intersections(ctx, a)
            o = np.argsort(g["idx"])
            assert np.array_equal(g["idx"][o], ref.idx[a])
            # the surface point lies r_p from the nearest free probe centre.  (The oracle's own roots stop
            # at 1e-11 of that distance, which the larger sizes' rounding does not reach.)
            p = origin + np.stack(np.unravel_index(g["idx"], dims), 1).astype(float)
            p[:, a] += g["tau"]
            d = oracle.distance(xyz, rad, r_p, p, 1.1 * r_p)[0]
            assert np.abs(d - r_p).max(initial=0.0) < TAU_TOL_A
    finally:
        eses.eses_destroy(ctx)


@pytest.mark.parametrize("prec", [eses.ESES_PREC_FP32_FILTERED, eses.ESES_PREC_FP64])
@pytest.mark.parametrize("unit", [0.1, 10.0, 100.0])
def test_a_molecule_in_other_units(unit, prec):
    """The same molecule with every length multiplied: the same labels and taus,
    and above an angstrom to the unit no more candidates than there (the
    margins shrink against the radii)."""
    libbuild.build()
    xyz, rad = inputs.protein_like(60, 17, inputs.PROTEIN_DENSITY)
    seen = []
    for u in (1.0, unit):
        ref = oracle.run(u * xyz, u * rad, 1.4 * u, 0.4 * u, 0.9 * u)
        ctx = eses.eses_create(u * xyz, u * rad, 1.4 * u, 0.4 * u, 0.9 * u)
        try:
            eses.eses_set_option(ctx, eses.ESES_OPT_PRECISION, prec)
            eses.eses_run(ctx)
            assert np.array_equal(eses.eses_labels(ctx), ref.labels)
            for a in range(3):
                g = eses.eses_intersections(ctx, a)
                o = np.argsort(g["idx"])
                assert np.array_equal(g["idx"][o], ref.idx[a])
                assert np.abs(g["tau"][o] - ref.tau[a]).max() * 0.4 < TAU_TOL_A
            st = eses.eses_stats(ctx)
            seen.append(st["sphere_candidates"] + st["torus_candidates"])
        finally:
            eses.eses_destroy(ctx)
    if unit > 1.0:
        assert seen[1] <= 1.01 * seen[0]
