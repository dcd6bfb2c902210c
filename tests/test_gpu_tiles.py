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


def _edges(lab):
    """Crossing edges per axis: 8x8x8 tiles in C order, then point order."""
    out = []
    for a in range(3):
        g = np.argwhere(np.diff(lab.astype(np.int16), axis=a) != 0)
        t, l = g // 8, g % 8
        nt = [-(-d // 8) for d in lab.shape]
        key = ((t[:, 0] * nt[1] + t[:, 1]) * nt[2] + t[:, 2]) * 512 + (l[:, 0] * 8 + l[:, 1]) * 8 + l[:, 2]
        g = g[np.argsort(key, kind="stable")]
        out.append((g[:, 0] * lab.shape[1] + g[:, 1]) * lab.shape[2] + g[:, 2])
    return out


@pytest.mark.parametrize("dims", [(1, 1, 1), (1, 1, 9), (3, 2, 5), (8, 8, 8), (9, 9, 9), (17, 8, 16), (7, 65, 33),
                                  (33, 130, 257), (160, 170, 300)])
@pytest.mark.parametrize("shift", [0, 1, 2, 3])
def test_noalloc_rows_at_every_alignment(dims, shift):
    """Label rows at every alignment of the first label and of a row (odd
    lengths), grids smaller than a word, one and several tiles per warp."""
    import torch

    libbuild.build()
    rng = np.random.default_rng(sum(dims) + shift)
    lab = (rng.random(dims) < 0.4).astype(np.int8)
    if max(dims) > 100:
        lab[: dims[0] // 2] = 1  # whole tiles without edges
    store = torch.full((lab.size + shift,), 1, dtype=torch.int8, device="cuda")
    store[shift:] = torch.from_numpy(lab.reshape(-1)).cuda()
    ref = _edges(lab)
    outs = [torch.full((len(r) + 1,), -1, dtype=torch.int64, device="cuda") for r in ref]
    counts = eses.eses_crossing_edges_noalloc(store.data_ptr() + shift, dims, *outs, [len(r) for r in ref])
    for a in range(3):
        assert counts[a] == len(ref[a])
        got = outs[a].cpu().numpy()
        assert np.array_equal(got[:-1], ref[a]) and got[-1] == -1, a


@pytest.mark.parametrize("prec", [eses.ESES_PREC_FP32_FILTERED, eses.ESES_PREC_FP64])
@pytest.mark.parametrize("h,r_p", [(0.2, 1.4), (0.45, 0.3), (0.95, 1.4), (0.5, 4.0), (3.9, 1.4), (4.1, 1.4), (12.0, 0.4)])
def test_torus_roots_from_short_to_long_edges(h, r_p, prec):
    """Edges from a seventh of the probe to past the molecule, tori from thin ones to
    those that meet themselves: every root next to the oracle's."""
    libbuild.build()
    xyz, rad = inputs.protein_like(30, 91, inputs.PROTEIN_DENSITY)
    margin = 1.5 * h + 0.3
    ref = oracle.run(xyz, rad, r_p, h, margin)
    ctx = eses.eses_create(xyz, rad, r_p, h, margin)
    try:
        eses.eses_set_option(ctx, eses.ESES_OPT_PRECISION, prec)
        eses.eses_run(ctx)
        assert np.array_equal(eses.eses_labels(ctx), ref.labels)
        for a in range(3):
            g = eses.eses_intersections(ctx, a)
            o = np.argsort(g["idx"])
            assert np.array_equal(g["idx"][o], ref.idx[a])
            assert np.abs(g["tau"][o] - ref.tau[a]).max() * h < 1e-6
    finally:
        eses.eses_destroy(ctx)


def test_circle_with_many_free_end_points():
    """Two large balls whose circle carries 35 small ones, none touching the
    next: 70 free triple points on one circle, more than the arc kernel lists
    for one thread each, so the circle is emitted whole by a warp."""
    libbuild.build()
    rho = np.sqrt((30.0 + 1.4) ** 2 - 10.0 ** 2)
    phi = 2.0 * np.pi * np.arange(35) / 35
    ring = np.stack([np.zeros(35), rho * np.cos(phi), rho * np.sin(phi)], 1)
    xyz = np.concatenate([[[-10.0, 0.0, 0.0], [10.0, 0.0, 0.0]], ring])
    rad = np.concatenate([[30.0, 30.0], np.full(35, 0.5)])
    ref = oracle.run(xyz, rad, 1.4, 1.5, 1.6)
    ctx = eses.eses_create(xyz, rad, 1.4, 1.5, 1.6)
    try:
        eses.eses_set_option(ctx, eses.ESES_OPT_GRAPH, 1)
        for _ in range(3):  # planned, captured, replayed
            eses.eses_run(ctx)
            patch = eses.eses_patch_data(ctx)
            v = patch["vertices"]
            # every triple point on both large spheres and on one small one
            d = np.linalg.norm(v[:, None, :] - xyz[None], axis=2) - (rad + 1.4)
            assert np.abs(d[:, :2]).max() < 1e-9 and np.abs(d[:, 2:]).min(1).max() < 1e-9
            assert len(v) == 70
            assert np.array_equal(eses.eses_labels(ctx), ref.labels)
            for a in range(3):
                g = eses.eses_intersections(ctx, a)
                o = np.argsort(g["idx"])
                assert np.array_equal(g["idx"][o], ref.idx[a])
                assert np.abs(g["tau"][o] - ref.tau[a]).max() * 1.5 < 1e-6
    finally:
        eses.eses_destroy(ctx)


@pytest.mark.parametrize("k", [2, 3, 5, 8, 31, 32, 33, 40])
def test_circle_covered_all_around(k):
    """The circle of two large balls under a ring of k others: neighbours that
    miss each other by a thousandth leave two free triple points each, that
    overlap by a thousandth none, and two where one of the ring is missing."""
    libbuild.build()
    rho = np.sqrt((30.0 + 1.4) ** 2 - 10.0 ** 2)
    phi = 0.3 + 2.0 * np.pi * np.arange(k) / k
    for delta, drop, expect in ((-1e-3, 0, 2 * k), (1e-3, 0, 0), (1e-3, 1, 2)):
        ring = np.stack([np.zeros(k), rho * np.cos(phi), rho * np.sin(phi)], 1)[drop:]
        reach = 2.0 * rho * np.sin(0.5 * np.pi / k * (1.0 + delta))  # covers pi / k (1 + delta) to either side
        xyz = np.concatenate([[[-10.0, 0.0, 0.0], [10.0, 0.0, 0.0]], ring])
        rad = np.concatenate([[30.0, 30.0], np.full(k - drop, reach - 1.4)])
        ctx = eses.eses_create(xyz, rad, 1.4, 3.0, 3.1)
        try:
            eses.eses_run(ctx)
            v = eses.eses_patch_data(ctx)["vertices"]
            d = np.abs(np.linalg.norm(v[:, None, :] - xyz[None, :2], axis=2) - 31.4) if len(v) else np.zeros((0, 2))
            assert int((d.max(1) < 1e-9).sum() if len(d) else 0) == expect
        finally:
            eses.eses_destroy(ctx)


def test_buffers_left_by_grown_ones_are_taken_again():
    """Runs of changing size in one context (block selections up and down, the
    whole grid) reuse the memory they gave up: after the first round the
    device's free memory stays where it is, the results stay the same, and
    destroying the context gives everything back."""
    import torch

    libbuild.build()
    torch.cuda.synchronize()
    free0, _ = torch.cuda.mem_get_info()
    xyz, rad = inputs.protein_like(600, 4, inputs.PROTEIN_DENSITY)
    ctx = eses.eses_create(xyz, rad, 1.4, 0.3, 0.8)
    try:
        eses.eses_set_option(ctx, eses.ESES_OPT_BLOCK_PTS, 16)
        nb = eses.eses_num_blocks(ctx)
        seen, free = {}, []
        for cycle in range(4):
            for cut in (1, int(nb[0]), 2, int(nb[0]) - 1, None):
                if cut is None:
                    eses.eses_set_blocks(ctx)
                else:
                    eses.eses_set_blocks(ctx, [0, 0, 0], [cut, int(nb[1]), int(nb[2])])
                eses.eses_run(ctx)
                got = (eses.eses_labels(ctx).tobytes(), *[eses.eses_intersections(ctx, a)["idx"].tobytes()
                                                          for a in range(3)], eses.eses_area_volume(ctx))
                assert seen.setdefault(cut, got) == got
            free.append(torch.cuda.mem_get_info()[0])
        assert free[1:] == free[1:2] * 3
    finally:
        eses.eses_destroy(ctx)
    torch.cuda.synchronize()
    free1, _ = torch.cuda.mem_get_info()
    assert abs(free1 - free0) <= 1 << 20
