"""The FP32 form's list of roots that FP64 must decide."""
import numpy as np
import pytest

import oracle
from paper_1809_04352_gb300 import build as libbuild
from paper_1809_04352_gb300 import eses, inputs

pytestmark = pytest.mark.gpu


def test_more_fp64_roots_than_first_planned():
    """A molecule next to a ball of 900, which sets the bound of staged FP32
    differences to half a thousandth, so that FP32 decides hardly any saddle root:
    the list outgrows its first size, the launches run again with a longer
    one, and the edges that lacked roots meanwhile are no failures.  The second
    and third runs are captured and replayed."""
    libbuild.build()
    xyz, rad = inputs.protein_like(300, 23, inputs.PROTEIN_DENSITY)
    xyz, rad, h = 10.0 * xyz, 10.0 * rad, 4.0
    dims, lo = oracle.grid(xyz, rad, h, 9.0)
    xyz = np.concatenate([xyz, xyz.max(0, keepdims=True) + 2000.0])
    rad = np.append(rad, 900.0)
    ref = oracle.run_on_grid(xyz, rad, 14.0, h, lo, dims)
    n = sum(len(i) for i in ref.idx)
    ctx = eses.eses_create_on_grid(xyz, rad, 14.0, h, lo, dims)
    try:
        eses.eses_set_option(ctx, eses.ESES_OPT_GRAPH, 1)
        for _ in range(3):
            eses.eses_run(ctx)
            st = eses.eses_stats(ctx)
            assert st["root_failures"] == 0
            assert st["torus_candidates"] > 1.2 * n + 4352  # the first size is the edges and 4,352
            assert np.array_equal(eses.eses_labels(ctx), ref.labels)
            for a in range(3):
                g = eses.eses_intersections(ctx, a)
                o = np.argsort(g["idx"])
                assert np.array_equal(g["idx"][o], ref.idx[a])
                assert np.abs(g["tau"][o] - ref.tau[a]).max() * h < 1e-6
    finally:
        eses.eses_destroy(ctx)
