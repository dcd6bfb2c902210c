"""Surface points that lie exactly on grid points: the edge that ends there
has its root at 0 or h, to the last bit or beside it by rounding."""
import numpy as np
import pytest

import oracle
from paper_1809_04352_gb300 import build as libbuild
from paper_1809_04352_gb300 import eses

pytestmark = pytest.mark.gpu

TAU_TOL_A = 1e-6  # the root tolerance of every comparison with the oracle


def _compare(ctx, ref, h):
    eses.eses_run(ctx)
    assert np.array_equal(eses.eses_labels(ctx), ref.labels)
    for a in range(3):
        g = eses.eses_intersections(ctx, a)
        o = np.argsort(g["idx"])
        assert np.array_equal(g["idx"][o], ref.idx[a])
        assert np.abs(g["tau"][o] - ref.tau[a]).max(initial=0.0) * h < TAU_TOL_A
    assert eses.eses_stats(ctx)["root_failures"] == 0


@pytest.mark.parametrize("prec", [eses.ESES_PREC_FP32_FILTERED, eses.ESES_PREC_FP64])
@pytest.mark.parametrize("axes", [(0, 1, 2), (1, 2, 0), (2, 0, 1)])
def test_saddle_and_spheres_through_grid_points(axes, prec):
    """Two balls of 1.25 at +-2 and a probe of 1.25 on a grid of 0.25: the
    saddle passes through (0.5, 0, 0.75) and the balls through (0.75, 1, 2),
    all grid points, and so do their images."""
    libbuild.build()
    xyz = np.array([[0.0, 0.0, -2.0], [0.0, 0.0, 2.0]])[:, list(axes)]
    rad = np.array([1.25, 1.25])
    ref = oracle.run(xyz, rad, 1.25, 0.25, 1.0)
    for a in range(3):  # ends of edges of both patches, from inside and from outside
        for k in (0, 1):
            assert (np.abs(ref.tau[a][ref.ptype[a] == k]) < 1e-9).any()
            assert (np.abs(ref.tau[a][ref.ptype[a] == k] - 1.0) < 1e-9).any()
    ctx = eses.eses_create(xyz, rad, 1.25, 0.25, 1.0)
    try:
        eses.eses_set_option(ctx, eses.ESES_OPT_PRECISION, prec)
        _compare(ctx, ref, 0.25)
    finally:
        eses.eses_destroy(ctx)


@pytest.mark.parametrize("prec", [eses.ESES_PREC_FP32_FILTERED, eses.ESES_PREC_FP64])
def test_saddle_root_on_a_grid_point_before_a_later_exit(prec):
    """An edge whose inside end point lies on the saddle, with a third ball's
    surface further along it: the root is the end point, not that exit.  (The
    plane y = 0 only: lines along y touch the saddle there.)"""
    libbuild.build()
    h = 2.375
    xyz = np.array([[0.0, 0.0, -2.0], [0.0, 0.0, 2.0], [3.0, 0.0, -0.375]])
    rad = np.array([1.875, 1.875, 0.25])
    dims = np.array([6, 1, 6])
    lo = np.array([1.0, 0.0, -0.375]) - h * np.array([2.0, 0.0, 2.0])
    ref = oracle.run_on_grid(xyz, rad, 0.625, h, lo, dims)
    at = (2 * 1 + 0) * 6 + 2  # the point (1, 0, -0.375)
    assert ref.tau[0][ref.idx[0] == at] == 0.0
    ctx = eses.eses_create_on_grid(xyz, rad, 0.625, h, lo, dims)
    try:
        eses.eses_set_option(ctx, eses.ESES_OPT_PRECISION, prec)
        _compare(ctx, ref, h)
    finally:
        eses.eses_destroy(ctx)
