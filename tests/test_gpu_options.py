"""Launch-shape options read back as what the runs take."""
import numpy as np
import pytest

from paper_1809_04352_gb300 import build as libbuild
from paper_1809_04352_gb300 import eses, inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("key", [eses.ESES_OPT_CLS_TILES, eses.ESES_OPT_EDGE_TILES])
def test_tiles_per_pop_reads_as_taken(key):
    """Single tiles until the option is set; the value that was set after that."""
    libbuild.build()
    xyz, rad = inputs.protein_like(30, 5, inputs.PROTEIN_DENSITY)
    ctx = eses.eses_create(xyz, rad, 1.4, 0.5, 0.9)
    try:
        assert eses.eses_get_option(ctx, key) == 1
        eses.eses_run(ctx)
        lab = eses.eses_labels(ctx)
        for v in (1, 7, 64):
            eses.eses_set_option(ctx, key, v)
            assert eses.eses_get_option(ctx, key) == v
            eses.eses_run(ctx)
            assert np.array_equal(eses.eses_labels(ctx), lab)
        for v in (0, 65):
            with pytest.raises(eses.EsesError):
                eses.eses_set_option(ctx, key, v)
            assert eses.eses_get_option(ctx, key) == 64
    finally:
        eses.eses_destroy(ctx)
