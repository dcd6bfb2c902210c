"""Launch shapes timed on a context whose cavities are filled."""
import numpy as np
import pytest

import oracle
from paper_1809_04352_gb300 import build as libbuild
from paper_1809_04352_gb300 import eses, inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [eses.ESES_PREC_FP32_FILTERED, eses.ESES_PREC_FP64])
def test_autotune_of_the_exterior_only_surface(prec):
    """Between its timings the autotuner classifies again, and the edge lists
    hold the filled labels' edges only: the fill is part of it.  Results after
    it as an untuned run's and the oracle's."""
    libbuild.build()
    xyz, rad = inputs.hollow_shell(shell_radius=6.5)
    ref = oracle.run(xyz, rad, 1.4, 0.5, 1.0, exterior=True)
    seen = []
    for tune in (False, True):
        ctx = eses.eses_create(xyz, rad, 1.4, 0.5, 1.0)
        try:
            eses.eses_set_option(ctx, eses.ESES_OPT_PRECISION, prec)
            eses.eses_set_option(ctx, eses.ESES_OPT_EXTERIOR, 1)
            if tune:
                eses.eses_autotune(ctx, 1)
            else:
                eses.eses_run(ctx)
            for _ in range(2):
                lab = eses.eses_labels(ctx)
                assert np.array_equal(lab, ref.labels)
                axes = []
                for a in range(3):
                    g = eses.eses_intersections(ctx, a)
                    o = np.argsort(g["idx"])
                    assert np.array_equal(g["idx"][o], ref.idx[a])
                    assert np.abs(g["tau"][o] - ref.tau[a]).max() * 0.5 < 1e-6
                    axes.append((g["idx"].tobytes(), g["tau"].tobytes(), g["normal"].tobytes()))
                seen.append((axes, eses.eses_area_volume(ctx), eses.eses_stats(ctx)["cavity_points"]))
                eses.eses_run(ctx)
        finally:
            eses.eses_destroy(ctx)
    assert all(s == seen[0] for s in seen)
