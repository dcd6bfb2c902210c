"""The work that users of this library have it do, as cases that can be timed
and compared.

A case is a dict of plain values; ``kind`` names the way the library is used:

  surface   one molecule from host atoms to host results, once
            (``eses.Surface``: create, run, read, close)
  step      a context that a program keeps and runs, results left in device
            memory (optionally FP64, with the tile proposer, replayed as a
            CUDA graph as the benchmark does)
  batch     the same for many molecules of uneven size in one context
  exterior  a kept context with the exterior-only surface (cavities filled)
  mesh      a kept context, run and turned into a triangle mesh on the host
  stream    a grid run slab by slab through ``stream.stream``
  train     one training step of the tile proposer (gradient and Adam)
  edges     the allocation-free crossing-edge listing of a device label grid

``prepare`` makes the inputs from the seed and what a program keeps (a
context, parameters, buffers for the results); ``run`` is one pass, its
results moved into those buffers, which are sized for any molecule of the
case's kind and size and hold zeros past the results; ``work`` the bytes and
flops no implementation can do without; ``exact`` plain 64-bit results for the
cases small enough for brute force.
"""
import functools
import math

import numpy as np
import torch

from paper_1809_04352_gb300 import eses, inputs, proposer
from paper_1809_04352_gb300 import stream as streaming

R_P = 1.4


def listed():
    return [
        # the smallest call: a ligand-sized fragment with the wrapper's defaults, where launches,
        # allocations and host reads are all there is
        {"name": "fragment-60", "kind": "surface", "shape": "globule", "atoms": 60, "r_p": R_P, "h": 0.5, "margin": 1.0},
        # the plain FP64 workload: 200 atoms of an open chain, every stage in FP64
        {"name": "plain-200", "kind": "step", "shape": "walk", "atoms": 200, "r_p": R_P, "h": 0.5, "margin": 4.0,
         "fp64": True, "proposer": False},
        # an ordinary molecule, once: what a script that goes through a list of structures does for each
        {"name": "surface-1501", "kind": "surface", "shape": "globule", "atoms": 1501, "r_p": R_P, "h": 0.4,
         "margin": 0.8},
        # the benchmark's headline step
        {"name": "globule-5000", "kind": "step", "shape": "globule", "atoms": 5000, "r_p": R_P, "h": 0.25,
         "margin": 0.8, "fp64": False, "proposer": True},
        # the largest call: a big complex on a fine grid (about 2e8 points)
        {"name": "globule-20000", "kind": "step", "shape": "globule", "atoms": 20000, "r_p": R_P, "h": 0.25,
         "margin": 0.8, "fp64": False, "proposer": True},
        # atoms packed as densely as in a crystal structure: most patches buried, the patch build weighs most
        {"name": "packed-5000", "kind": "step", "shape": "packed", "atoms": 5000, "r_p": R_P, "h": 0.25, "margin": 0.8,
         "fp64": False, "proposer": False},
        # a screening batch: molecules of uneven size in one context on a coarse grid
        {"name": "batch-32", "kind": "batch", "molecules": 32, "lo": 300, "hi": 3000, "r_p": R_P, "h": 0.5,
         "margin": 0.8},
        # the surface that a probe reaches from outside (cavity points become inside)
        {"name": "exterior-2003", "kind": "exterior", "shape": "globule", "atoms": 2003, "r_p": R_P, "h": 0.4,
         "margin": 0.8},
        # a triangle mesh for display or a boundary-element solver
        {"name": "mesh-3000", "kind": "mesh", "shape": "globule", "atoms": 3000, "r_p": R_P, "h": 0.4, "margin": 0.8},
        # a grid taken slab by slab with two contexts, as for grids larger than the device
        {"name": "stream-6000", "kind": "stream", "shape": "globule", "atoms": 6000, "r_p": R_P, "h": 0.35,
         "margin": 0.8, "slabs": 5},
        # the proposer's training step at its batch size
        {"name": "train-4096", "kind": "train", "samples": 4096},
        # crossing edges of a caller's label grid into a caller's buffers
        {"name": "edges-257x301x211", "kind": "edges", "d0": 257, "d1": 301, "d2": 211},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["surface", "surface", "step", "step", "step", "batch", "exterior", "mesh", "stream", "train",
                       "edges"])
    r_p = round(rng.uniform(1.2, 1.6), 2)
    h = round(rng.uniform(0.3, 0.6), 3)
    margin = round(rng.uniform(0.8, 1.6), 2)
    if kind == "train":
        return {"kind": kind, "samples": _log(rng, 200, 8192)}
    if kind == "edges":
        return {"kind": kind, "d0": _log(rng, 30, 400), "d1": _log(rng, 30, 400), "d2": _log(rng, 30, 400)}
    if kind == "batch":
        lo = _log(rng, 60, 600)
        return {"kind": kind, "molecules": _log(rng, 3, 32), "lo": lo, "hi": 5 * lo, "r_p": r_p,
                "h": round(rng.uniform(0.4, 0.6), 3), "margin": margin}
    if kind == "step":
        shape = rng.choice(["globule", "globule", "walk", "packed"])
        fp64 = rng.random() < 0.25
        hi = {"globule": 12000, "walk": 400, "packed": 5000}[shape]
        return {"kind": kind, "shape": shape, "atoms": _log(rng, 30, min(hi, 900) if fp64 else hi), "r_p": r_p, "h": h,
                "margin": margin, "fp64": fp64, "proposer": (not fp64) and rng.random() < 0.5}
    if kind == "stream":
        return {"kind": kind, "shape": "globule", "atoms": _log(rng, 800, 6000), "r_p": r_p, "h": h, "margin": margin,
                "slabs": rng.randint(2, 6)}
    return {"kind": kind, "shape": rng.choice(["globule", "globule", "packed"]), "atoms": _log(rng, 20, 4000),
            "r_p": r_p, "h": h, "margin": margin}


# --------------------------------------------------------------------------
# inputs
# --------------------------------------------------------------------------
@functools.lru_cache(maxsize=1)
def _packed_base():
    xyz, rad = inputs.paper_density(5000, 2200)
    order = np.argsort(np.einsum("ij,ij->i", xyz, xyz), kind="stable")
    return xyz[order], rad[order]


def _rotation(rng):
    q, r = np.linalg.qr(rng.standard_normal((3, 3)))
    q = q * np.sign(np.diag(r))
    return q if np.linalg.det(q) > 0 else -q


def _atoms(shape, n, seed):
    if shape == "globule":
        return inputs.protein_like(n, seed, inputs.PROTEIN_DENSITY)
    if shape == "walk":
        while True:  # an open chain; the few that are stretched past the result buffers are left out
            xyz, rad = inputs.protein_like(n, seed, None)
            if (xyz.max(0) - xyz.min(0)).max() <= _extent("walk", n):
                return xyz, rad
            seed += 1 << 32
    # the n atoms nearest the centre of a packed globule, turned and moved a little by the seed
    xyz, rad = _packed_base()
    rng = np.random.Generator(np.random.PCG64(seed))
    xyz = xyz[:n] @ _rotation(rng).T + rng.normal(0.0, 0.03, (n, 3))
    return np.ascontiguousarray(xyz), np.ascontiguousarray(rad[:n])


# --------------------------------------------------------------------------
# buffers for the results
# --------------------------------------------------------------------------
def _extent(shape, n):
    """Largest extent of the atom centres along an axis (A)."""
    if shape == "walk":
        return 12.0 + 4.0 * math.sqrt(n)
    density = inputs.PROTEIN_DENSITY if shape == "globule" else 0.08
    return 2.0 * max((3.0 * n / (4.0 * math.pi * density)) ** (1.0 / 3.0) - 2.5, inputs.STEP) + 6.0


def _room(shape, n, case):
    """Grid points, and crossing edges per axis, that any molecule of n atoms
    of this shape keeps within."""
    d = math.ceil((_extent(shape, n) + 3.7 + 2.0 * case["margin"]) / case["h"]) + 2
    area = 3.5 * (10.0 * n) ** (2.0 / 3.0) + 400.0 if shape == "packed" else 8.0 * n + 400.0
    return d ** 3, int(area / case["h"] ** 2)


_FIELDS = (("idx", 1, "int64"), ("tau", 1, "float64"), ("normal", 3, "float64"), ("tau32", 1, "float32"),
           ("normal32", 3, "float32"))


def _buffers(rooms, zeros, fields=_FIELDS):
    """One array per output for the molecules whose rooms are given."""
    points, edges = sum(r[0] for r in rooms), sum(r[1] for r in rooms)
    out = {"labels": zeros((points,), "int8"), "area_volume": np.zeros((len(rooms), 2))}
    for a in range(3):
        for key, w, kind in fields:
            out[f"{key}{a}"] = zeros((edges, w) if w > 1 else (edges,), kind)
    return out


def _on_device(shape, kind):
    return torch.zeros(shape, dtype=getattr(torch, kind), device="cuda")


def _batch(case, seed):
    sizes = inputs.batch_sizes(case["molecules"], case["lo"], case["hi"])
    return [inputs.protein_like(int(n), 1000 * (seed % 100003) + k, inputs.PROTEIN_DENSITY)
            for k, n in enumerate(sizes)]


class _Owner:
    """A library context, released once neither the program nor any view of
    its results is left."""

    def __init__(self, ctx):
        self.ctx = ctx

    def __del__(self):
        eses.eses_destroy(self.ctx)


class _Lent:
    """A device buffer that a context lends, for torch to view; the view keeps
    this object, and so the context."""

    def __init__(self, owner, ptr, shape, typestr):
        self.owner = owner
        self.__cuda_array_interface__ = {"data": (ptr, False), "shape": shape, "typestr": typestr, "version": 3}


class Context:
    """A context that a program keeps, and torch views of its device results
    (made again only when a buffer or its size has changed)."""

    def __init__(self, ctx):
        self.owner = _Owner(ctx)
        self.ctx = ctx
        self.n_mol = eses.eses_num_molecules(ctx)
        self.grids = [eses.eses_mol_grid(ctx, m)[0] for m in range(self.n_mol)]
        self.views = {}

    def view(self, name, ptr, shape, typestr):
        have = self.views.get(name)
        if have is None or have[0] != (ptr, shape):
            have = ((ptr, shape), torch.as_tensor(_Lent(self.owner, ptr, shape, typestr), device="cuda"))
            self.views[name] = have
        return have[1]

    def results(self, out):
        """Moves labels, intersections (per axis), areas and volumes into
        `out`: the molecules' results lie one after the other, from the first
        one's pointer to the end of the last one's."""
        last = self.n_mol - 1
        p0 = eses.eses_mol_labels_device(self.ctx, 0)
        n = eses.eses_mol_labels_device(self.ctx, last) + int(np.prod(self.grids[last])) - p0
        out["labels"][:n].copy_(self.view("labels", p0, (n,), "|i1"))
        for a in range(3):
            ptrs = eses.eses_mol_intersections_device(self.ctx, 0, a)
            n = eses.eses_mol_num_intersections(self.ctx, last, a)
            if last:
                n += (eses.eses_mol_intersections_device(self.ctx, last, a)[0] - ptrs[0]) // 8
            for (key, w, _), ptr, kind in zip(_FIELDS, ptrs, ("<i8", "<f8", "<f8", "<f4", "<f4")):
                if n:
                    key = f"{key}{a}"
                    out[key][:n].copy_(self.view(key, ptr, (n, w) if w > 1 else (n,), kind))
        for m in range(self.n_mol):
            out["area_volume"][m] = eses.eses_mol_area_volume(self.ctx, m)
        return out


@functools.lru_cache(maxsize=1)
def _params():
    return proposer.load_params()


def prepare(case, seed):
    kind = case["kind"]
    if kind == "train":
        return _prepare_train(case, seed)
    if kind == "edges":
        return _prepare_edges(case, seed)
    if kind == "batch":
        mols = _batch(case, seed)
        ctx = eses.eses_create_batch(mols, case["r_p"], case["h"], case["margin"])
        eses.eses_set_option(ctx, eses.ESES_OPT_GRAPH, 1)
        return case, Context(ctx), _buffers([_room("globule", len(r), case) for _, r in mols], _on_device)
    xyz, rad = _atoms(case["shape"], case["atoms"], seed)
    room = _room(case["shape"], case["atoms"], case)
    if kind == "surface":
        return case, (xyz, rad), _buffers([room], np.zeros)
    if kind == "stream":
        return case, (xyz, rad), _buffers([room], np.zeros, _FIELDS[:3])
    ctx = eses.eses_create(xyz, rad, case["r_p"], case["h"], case["margin"])
    if kind == "mesh":
        return case, Context(ctx), {"keys": np.zeros((6 * room[1], 3), np.int64), "xyz": np.zeros((6 * room[1], 3, 3)),
                                    "area_volume": np.zeros(2)}
    if kind == "step":
        eses.eses_set_option(ctx, eses.ESES_OPT_GRAPH, 1)
        if case["fp64"]:
            eses.eses_set_option(ctx, eses.ESES_OPT_PRECISION, eses.ESES_PREC_FP64)
        if case["proposer"]:
            eses.eses_set_proposer(ctx, eses.ESES_PROPOSER_MLP, _params(), 0.5)
    elif kind == "exterior":
        eses.eses_set_option(ctx, eses.ESES_OPT_EXTERIOR, 1)
    return case, Context(ctx), _buffers([room], _on_device)


def run(state):
    return _RUN[state[0]["kind"]](*state)


def _run_context(case, held, out):
    eses.eses_run(held.ctx)
    return held.results(out)


def _c(code, ctx):
    if code != eses.ESES_OK:
        raise eses.EsesError(code, eses.eses_last_error(ctx))


def _run_mesh(case, held, out):
    eses.eses_run(held.ctx)
    n = eses.eses_mesh_count(held.ctx)
    if n > len(out["keys"]):
        raise ValueError("the mesh does not fit its buffers")
    _c(eses.load().eses_mesh(held.ctx, out["keys"].ctypes.data, out["xyz"].ctypes.data), held.ctx)
    out["area_volume"][:] = eses.eses_area_volume(held.ctx)
    return out


def _run_surface(case, atoms, out):
    with eses.Surface(atoms[0], atoms[1], case["r_p"], case["h"], case["margin"]) as s:
        s.run()
        if int(np.prod(s.grid()[0])) > len(out["labels"]):
            raise ValueError("the labels do not fit their buffer")
        eses.eses_labels(s.ctx, out["labels"])
        for a in range(3):
            if eses.eses_num_intersections(s.ctx, a) > len(out[f"idx{a}"]):
                raise ValueError("the intersections do not fit their buffers")
            _c(eses.load().eses_intersections(s.ctx, a, *[out[f"{key}{a}"].ctypes.data for key, _, _ in _FIELDS]),
               s.ctx)
        out["area_volume"][0] = s.area_volume()
    return out


def _run_stream(case, atoms, out):
    dims = _dims(atoms[0], atoms[1], case)
    layer = 64 * dims[1] * dims[2]
    per = -(-(-(-dims[0] // 64)) // case["slabs"])  # block layers per slab
    parts = {}

    def sink(k, part):
        at = int(part.lo[0]) * dims[1] * dims[2]
        out["labels"][at:at + part.labels.size] = part.labels.reshape(-1)
        parts[k] = (part.idx, part.tau, part.normal)

    tot = streaming.stream(atoms[0], atoms[1], case["r_p"], case["h"], case["margin"], sink,
                           max_points=per * layer, block_pts=64)
    out["area_volume"][0] = tot["area"], tot["volume"]
    for a in range(3):
        n = 0
        for k in sorted(parts):
            m = n + len(parts[k][0][a])
            for (key, _, _), v in zip(_FIELDS, parts[k]):
                out[f"{key}{a}"][n:m] = v[a]
            n = m
    return out


# the proposer's training data: features as the library makes them (log counts, a position in [0, 1], a size
# ratio) and targets that follow the density, class-balanced weights
def _prepare_train(case, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    n = case["samples"]
    dens = torch.rand((n, 1), generator=g, device="cuda") * 6.0
    x = torch.empty((n, 32), device="cuda")
    x[:, :27] = torch.log1p(torch.floor(torch.rand((n, 27), generator=g, device="cuda") * dens))
    x[:, 27:30] = torch.rand((n, 3), generator=g, device="cuda")
    x[:, 30] = torch.log1p(torch.expm1(x[:, :27]).sum(1))
    x[:, 31] = 0.26
    y = (x[:, 13] + 0.2 * x[:, 30] + 0.1 * torch.randn(n, generator=g, device="cuda") > 1.2).float()
    pos = y.sum().clamp(min=1.0)
    w = torch.where(y > 0, 0.5 / pos, 0.5 / (n - pos).clamp(min=1.0))
    p = torch.from_numpy(proposer.init_params(seed)).cuda()
    m = 1e-3 * torch.randn(p.shape, generator=g, device="cuda")
    v = 1e-6 * torch.rand(p.shape, generator=g, device="cuda")
    return case, None, {"x": x.contiguous(), "y": y, "w": w.contiguous(), "p0": p, "m0": m, "v0": v,
                  "p": torch.empty_like(p), "m": torch.empty_like(m), "v": torch.empty_like(v),
                  "grad": torch.empty_like(p), "loss": torch.empty(1, device="cuda"),
                  "scratch": torch.empty(eses.eses_mlp_grad_scratch(n), device="cuda")}


_STEP, _LR = 3, 2e-3


def _run_train(case, _, d):
    stream = torch.cuda.current_stream().cuda_stream
    # the step updates in place; it starts from the same state on every pass
    torch._foreach_copy_([d["p"], d["m"], d["v"]], [d["p0"], d["m0"], d["v0"]])
    eses.eses_mlp_grad(d["x"], d["y"], d["w"], case["samples"], d["p"], d["grad"], d["loss"], d["scratch"], stream)
    eses.eses_mlp_adam(d["p"], d["grad"], d["m"], d["v"], _STEP, _LR, stream)
    return {k: d[k] for k in ("grad", "loss", "p", "m", "v")}


def _edge_room(dims):
    return int(0.15 * dims[0] * dims[1] * dims[2]) + 1000


# labels of a smooth closed shape: waves of about the size of a side chain inside a ball
def _prepare_edges(case, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    dims = (case["d0"], case["d1"], case["d2"])
    ax = [torch.arange(d, device="cuda", dtype=torch.float32) for d in dims]
    f = torch.zeros(dims, device="cuda")
    k = torch.randn((6, 3), generator=g, device="cuda") * 0.12
    ph = torch.rand(6, generator=g, device="cuda") * 6.28
    for j in range(6):
        f += torch.cos(k[j, 0] * ax[0][:, None, None] + k[j, 1] * ax[1][None, :, None] + k[j, 2] * ax[2][None, None, :]
                       + ph[j])
    r2 = sum((((a - 0.5 * (d - 1)) / (0.5 * d - 1)) ** 2).view([-1 if i == q else 1 for q in range(3)])
             for i, (a, d) in enumerate(zip(ax, dims)))
    labels = ((f > -0.5) & (r2 < 0.95)).to(torch.int8).contiguous()
    cap = _edge_room(dims)
    return case, None, {"labels": labels, "dims": dims, "cap": [cap] * 3,
                        "out": [torch.zeros(cap, dtype=torch.int64, device="cuda") for _ in range(3)]}


def _run_edges(case, _, d):
    stream = torch.cuda.current_stream().cuda_stream
    counts = eses.eses_crossing_edges_noalloc(d["labels"], d["dims"], *d["out"], d["cap"], stream)
    return {"counts": counts, "idx": d["out"]}


_RUN = {"surface": _run_surface, "step": _run_context, "batch": _run_context, "exterior": _run_context,
        "mesh": _run_mesh, "stream": _run_stream, "train": _run_train, "edges": _run_edges}


# --------------------------------------------------------------------------
# the work of a pass
# --------------------------------------------------------------------------
def _dims(xyz, rad, case):
    lo = (xyz - rad[:, None]).min(0) - case["margin"]
    hi = (xyz + rad[:, None]).max(0) + case["margin"]
    return [int(math.ceil((b - a) / case["h"])) + 1 for a, b in zip(lo, hi)]


# crossing edges times h^2 per atom (1.5 times the surface area per atom) and flops per grid point (each point
# against the atoms that reach it, each shell point against its candidate patches), by the kind of molecule
_EDGE_AREA = {"globule": 14.2, "walk": 23.0, "packed": 1.6}
_POINT_FLOPS = {"globule": 119.0, "walk": 40.0, "packed": 500.0}
_EDGE_FLOPS = 1000.0


def _surface_work(shape, xyz, rad, case):
    points = float(np.prod(np.array(_dims(xyz, rad, case), dtype=np.float64)))
    edges = _EDGE_AREA[shape] * len(rad) / case["h"] ** 2
    return 32.0 * len(rad) + points + 56.0 * edges, _POINT_FLOPS[shape] * points + _EDGE_FLOPS * edges, edges


def work(case):
    kind = case["kind"]
    if kind == "train":
        n, p = case["samples"], eses.ESES_MLP_NPARAM
        return {"bytes": 4.0 * (34 * n + 7 * p), "flops": 6.0 * p * n}
    if kind == "edges":
        points = float(case["d0"]) * case["d1"] * case["d2"]
        return {"bytes": points + 8.0 * 0.08 * points, "flops": 3.0 * points}
    if kind == "batch":
        tot = [_surface_work("globule", x, r, case) for x, r in _batch(case, 0)]
        return {"bytes": sum(t[0] for t in tot), "flops": sum(t[1] for t in tot)}
    xyz, rad = _atoms(case["shape"], case["atoms"], 0)
    nbytes, flops, edges = _surface_work(case["shape"], xyz, rad, case)
    if kind == "mesh":
        # about two triangles to a vertex (one vertex per crossing edge), 96 bytes each
        nbytes = 32.0 * len(rad) + 2.0 * edges * 96.0
    return {"bytes": nbytes, "flops": flops}


# --------------------------------------------------------------------------
# plain 64-bit results
# --------------------------------------------------------------------------
def exact(case, seed):
    if case["kind"] == "train":
        return _exact_train(case, seed)
    if case["kind"] in ("surface", "step") and case["atoms"] <= 260:
        xyz, rad = _atoms(case["shape"], case["atoms"], seed)
        return _Exact(xyz, rad, case).results(_room(case["shape"], case["atoms"], case)[1])
    return None


def _exact_train(case, seed):
    d = _prepare_train(case, seed)[2]
    x, y, w = (d[k].double() for k in ("x", "y", "w"))
    p = d["p0"].double().requires_grad_(True)
    w1, b1, w2, b2, w3, b3 = torch.split(p, [2048, 64, 4096, 64, 64, 1])
    h1 = torch.relu(x @ w1.view(32, 64) + b1)
    h2 = torch.relu(h1 @ w2.view(64, 64) + b2)
    z = h2 @ w3 + b3
    loss = (w * torch.nn.functional.binary_cross_entropy_with_logits(z, y, reduction="none")).sum()
    (g,) = torch.autograd.grad(loss, p)
    m = 0.9 * d["m0"].double() + 0.1 * g
    v = 0.999 * d["v0"].double() + 0.001 * g * g
    mh, vh = m / (1 - 0.9 ** _STEP), v / (1 - 0.999 ** _STEP)
    return {"grad": g, "loss": loss.detach().view(1), "p": p.detach() - _LR * mh / (vh.sqrt() + 1e-8), "m": m, "v": v}


class _Exact:
    """Brute force over all atoms, circles and triple points: the distance to
    the free probe centres, the first root of distance = r_p along every edge
    whose end labels differ, the unit normal and the estimators."""

    def __init__(self, xyz, rad, case):
        dev = "cuda" if torch.cuda.is_available() else "cpu"
        self.dev, self.rp, self.h = dev, case["r_p"], case["h"]
        self.lo = torch.tensor((xyz - rad[:, None]).min(0) - case["margin"], device=dev)
        self.dims = _dims(xyz, rad, case)
        self.c = torch.tensor(xyz, device=dev)
        self.r = torch.tensor(rad, device=dev)
        self.R = self.r + self.rp
        n = len(rad)
        d = torch.cdist(self.c, self.c, compute_mode="donot_use_mm_for_euclid_dist")
        i, j = torch.triu_indices(n, n, 1, device=dev)
        s = d[i, j]
        ok = (s < self.R[i] + self.R[j]) & (s > (self.R[i] - self.R[j]).abs())
        i, j, s = i[ok], j[ok], s[ok]
        self.u = (self.c[j] - self.c[i]) / s[:, None]
        t = (s * s + self.R[i] ** 2 - self.R[j] ** 2) / (2 * s)
        self.o = self.c[i] + t[:, None] * self.u
        self.rho = (self.R[i] ** 2 - t * t).clamp(min=0).sqrt()
        self.pi, self.pj = i, j
        # free triple points: each circle against every third sphere
        vs = []
        for k0 in range(0, len(i), 512):
            o, u, rho = (v[k0:k0 + 512] for v in (self.o, self.u, self.rho))
            a, b = self.pi[k0:k0 + 512], self.pj[k0:k0 + 512]
            q = self.c[None] - o[:, None]
            z = (q * u[:, None]).sum(-1)
            w = q - z[..., None] * u[:, None]
            wn = w.norm(dim=-1)
            # |rho cos - wn|^2 + (rho sin)^2 + z^2 = R_k^2
            cosv = (rho[:, None] ** 2 + wn ** 2 + z ** 2 - self.R[None] ** 2) / (2 * rho[:, None] * wn).clamp(min=1e-300)
            k = torch.arange(n, device=dev)[None]
            m = (cosv.abs() < 1) & (k > b[:, None]) & (wn > 1e-9)
            e, kk = torch.nonzero(m, as_tuple=True)
            e1 = w[e, kk] / wn[e, kk][:, None]
            e2 = torch.linalg.cross(u[e], e1)
            cs = cosv[e, kk]
            sn = (1 - cs * cs).sqrt()
            for sg in (1.0, -1.0):
                p = o[e] + rho[e][:, None] * (cs[:, None] * e1 + sg * sn[:, None] * e2)
                if len(p):
                    vs.append(p[self._free(p, torch.stack([a[e], b[e], kk], 1))])
        self.v = torch.cat(vs) if vs else torch.zeros((0, 3), dtype=torch.float64, device=dev)

    def _free(self, p, own):
        d = torch.cdist(p, self.c, compute_mode="donot_use_mm_for_euclid_dist") - self.R[None]
        d.scatter_(1, own, math.inf)
        return (d > -1e-9).all(1)

    def nearest(self, x):
        """Distance of x to the free probe centres, as far as it is below
        r_p + 2 h (else +inf), and the nearest free point."""
        best = torch.full((len(x),), math.inf, dtype=torch.float64, device=self.dev)
        wit = torch.zeros_like(x)
        dc = torch.cdist(x, self.c, compute_mode="donot_use_mm_for_euclid_dist")
        zero = (dc >= self.R[None]).all(1)
        reach = self.rp + 2 * self.h

        def take(e, p, own, dist):
            ok = self._free(p, own) if own is not None else torch.ones(len(p), dtype=torch.bool, device=self.dev)
            e, p, dist = e[ok], p[ok], dist[ok]
            new = best.scatter_reduce(0, e, dist, "amin")
            hit = dist == new[e]
            better = hit & (dist < best[e])
            wit[e[better]] = p[better]
            best.copy_(new)

        e, i = torch.nonzero((dc < self.R[None]) & (self.R[None] - dc < reach) & (dc > 0), as_tuple=True)
        take(e, self.c[i] + (x[e] - self.c[i]) * (self.R[i] / dc[e, i])[:, None], i[:, None], self.R[i] - dc[e, i])
        for k0 in range(0, len(self.o), 1024):
            o, u, rho = (v[k0:k0 + 1024] for v in (self.o, self.u, self.rho))
            q = x[:, None] - o[None]
            z = (q * u[None]).sum(-1)
            w = q - z[..., None] * u[None]
            wn = w.norm(dim=-1)
            dist = ((wn - rho[None]) ** 2 + z * z).sqrt()
            e, k = torch.nonzero((dist < reach) & (wn > 1e-12), as_tuple=True)
            p = o[k] + w[e, k] * (rho[k] / wn[e, k])[:, None]
            take(e, p, torch.stack([self.pi[k0 + k], self.pj[k0 + k]], 1), dist[e, k])
        dv = torch.cdist(x, self.v, compute_mode="donot_use_mm_for_euclid_dist")
        e, k = torch.nonzero(dv < reach, as_tuple=True)
        take(e, self.v[k], None, dv[e, k])
        best[zero] = 0.0
        return best, wit

    def results(self, room):
        d0, d1, d2 = self.dims
        h = self.h
        k = torch.arange(d0 * d1 * d2, device=self.dev)
        lab = torch.zeros(len(k), dtype=torch.bool, device=self.dev)
        for a in range(0, len(k), 1 << 17):
            q = k[a:a + (1 << 17)]
            x = self.point(q)
            dc = torch.cdist(x, self.c, compute_mode="donot_use_mm_for_euclid_dist")
            lab[q] = (dc <= self.r[None]).any(1)
            shell = torch.nonzero(~lab[q] & (dc < self.R[None]).any(1))[:, 0]
            for b in range(0, len(shell), 4096):
                s = shell[b:b + 4096]
                lab[q[s]] = self.nearest(x[s])[0] >= self.rp
        grid = lab.view(d0, d1, d2)
        out = {"labels": None}
        area = inside = 0.0
        for a in range(3):
            n = self.dims[a] - 1
            lo, hi = grid.narrow(a, 0, n), grid.narrow(a, 1, n)
            inside += float((lo & hi).sum()) * h
            at = torch.nonzero(lo != hi)
            t, l = at // 8, at % 8
            tiles = [-(-d // 8) for d in self.dims]
            key = ((t[:, 0] * tiles[1] + t[:, 1]) * tiles[2] + t[:, 2]) * 512 + (l[:, 0] * 8 + l[:, 1]) * 8 + l[:, 2]
            at = at[torch.argsort(key)]
            idx = (at[:, 0] * d1 + at[:, 1]) * d2 + at[:, 2]
            tau, nrm = self.roots(idx, a, lab[idx])
            area += h * h * float(nrm[:, a].abs().sum())
            inside += float(torch.where(lab[idx], tau, 1 - tau).sum()) * h
            out[f"idx{a}"] = None
            pad = torch.zeros((room - len(tau), 4), dtype=torch.float64, device=self.dev)
            out[f"tau{a}"] = out[f"tau32{a}"] = torch.cat([tau, pad[:, 0]])
            out[f"normal{a}"] = out[f"normal32{a}"] = torch.cat([nrm, pad[:, 1:]])
        out["area_volume"] = np.array([[area, h * h / 3 * inside]])
        return out

    def point(self, q):
        d0, d1, d2 = self.dims
        ijk = torch.stack([q // (d1 * d2), q // d2 % d1, q % d2], 1).double()
        return self.lo[None] + self.h * ijk

    def roots(self, idx, axis, inside):
        """First root of distance = r_p from the lower end: steps of |g| (g is
        1-Lipschitz, so no root is passed), Newton's step (the slope of the
        distance is that to the witness) near a root that crosses the way this one does."""
        taus, nrms = [], []
        for b in range(0, len(idx), 4096):
            x0 = self.point(idx[b:b + 4096])
            up = inside[b:b + 4096]
            t = torch.zeros(len(x0), dtype=torch.float64, device=self.dev)
            live = torch.arange(len(x0), device=self.dev)
            wit = torch.zeros_like(x0)
            for it in range(2000):
                x = x0[live].clone()
                x[:, axis] += t[live]
                dist, w = self.nearest(x)
                g = (dist - self.rp).clamp(max=self.h)
                slope = (x[:, axis] - w[:, axis]) / dist.clamp(min=1e-9)
                cross = torch.where(up[live], -slope, slope)
                newton = (g.abs() < 0.3 * cross ** 2) & (cross > 1e-5) & (dist > 0)
                s = torch.where(newton, -g / slope, torch.where(up[live], g.clamp(min=0), (-g).clamp(min=0)))
                wit[live] = w
                t[live] = (t[live] + s).clamp(0.0, self.h)
                live = live[(g.abs() > 1e-14) & (s.abs() > 1e-15)]
                if not len(live):
                    break
            x = x0.clone()
            x[:, axis] += t
            v = wit - x
            taus.append(t / self.h)
            nrms.append(v / v.norm(dim=1, keepdim=True))
        return torch.cat(taus), torch.cat(nrms)
