"""Kernels that work on tiles, at the sizes where their splits change."""
import numpy as np
import pytest

import oracle
from paper_1809_04352_gb300 import build as libbuild
from paper_1809_04352_gb300 import eses, inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [eses.ESES_PREC_FP32_FILTERED, eses.ESES_PREC_FP64])
@pytest.mark.parametrize("h", [0.15, 0.3, 0.9])
@pytest.mark.parametrize("n", [1, 2, 3, 9, 40])
def test_shell_points_of_few_and_many_lanes(n, h, prec):
    """From tiles with a handful of shell points (32 lanes share one) to tiles
    full of them (one lane each): labels as the oracle's."""
    libbuild.build()
    xyz, rad = inputs.protein_like(n, 60 + n, inputs.PROTEIN_DENSITY)
    ref = oracle.run(xyz, rad, 1.4, h, 0.9)
    ctx = eses.eses_create(xyz, rad, 1.4, h, 0.9)
    try:
        eses.eses_set_option(ctx, eses.ESES_OPT_PRECISION, prec)
        eses.eses_run(ctx)
        assert np.array_equal(eses.eses_labels(ctx), ref.labels)
    finally:
        eses.eses_destroy(ctx)

