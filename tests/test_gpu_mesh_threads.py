"""The first mesh of a context needs its case table on the device before the
kernels read it, whatever other threads and contexts do."""
import threading

import numpy as np
import pytest

from paper_1809_04352_gb300 import build as libbuild
from paper_1809_04352_gb300 import eses, inputs

import oracle
from oracle import mesh_oracle as mo

pytestmark = pytest.mark.gpu


def test_first_meshes_of_contexts_on_several_threads():
    """Four threads, each with contexts of its own made, run, meshed and
    destroyed: every mesh is the oracle's."""
    from tests.test_mesh import canonical

    libbuild.build()
    mols = [inputs.protein_like(n, 40 + n, inputs.PROTEIN_DENSITY) for n in (5, 20, 45, 80)]
    refs = []
    for xyz, rad in mols:
        r = oracle.run(xyz, rad, 1.4, 0.5, 0.9)
        refs.append(canonical(*mo.mesh(r.labels, r.lo, r.h, r.idx, r.tau)))
    start, bad = threading.Barrier(len(mols)), []

    def work(k):
        try:
            start.wait(60)
            for _ in range(12):
                ctx = eses.eses_create(*mols[k], 1.4, 0.5, 0.9)
                try:
                    eses.eses_run(ctx)
                    for _ in range(2):
                        keys, xyz = canonical(*eses.eses_mesh(ctx))
                        assert np.array_equal(keys, refs[k][0])
                        assert np.abs(xyz - refs[k][1]).max() < 1e-6
                finally:
                    eses.eses_destroy(ctx)
        except BaseException as e:  # reported by the test's own thread
            bad.append((k, repr(e)))

    threads = [threading.Thread(target=work, args=(k,)) for k in range(len(mols))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad
