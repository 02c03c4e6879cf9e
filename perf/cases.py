"""Workloads that this library is timed on, through its public Python calls.

Each case is a dict of plain values; ``prepare`` makes its inputs from a seed
(and what a program keeps between calls: the uploaded lattice, the batch's
plan, the buffers that the results are copied to), ``run`` does one pass,
``work`` says what a pass cannot do without and ``exact`` gives the outputs
that have a value in 64 bits.

Kinds of a case:

- ``slice``: layers of a lattice to contours, the call that the library exists
  for: a whole part whose contours stay on the device, or (``host``) a small
  part or one layer at a time, as a printer that streams its slices asks for
  them, in host memory;
- ``part``: the same from host arrays to page-locked host buffers, upload
  included (a part that is sliced once);
- ``mask``: the binary images of a whole part on the device, no contours (a
  DLP printer's input);
- ``field``: the field itself on a few layers beside the images, for programs
  that do their own extraction;
- ``tune``: one step of radius tuning through autograd: update, volume
  fraction of the cells, and its gradients;
- ``batch``: many small parts planned once and run as one graph, their
  contours taken;
- ``finish``: simplification, smoothing and infill of contours on the device;
- ``design``: vertex re-positioning and density matching of a tetrahedral
  mesh, host mesh in and host lattice out;
- ``depth``: a depth image of the solid.

Lattices: ``grid`` is a jittered Freudenthal grid (supports of 10 to 26
pixels), ``cells`` a cubic + body-centred lattice, ``graded`` an octree-graded
Freudenthal lattice of fine struts (supports of under 4 pixels, the largest
parts).

Contours, meshes and infill have as many entries as the inputs make them have;
a program copies them to buffers of its own, with room to spare, and so do the
passes here (the rest of a buffer stays 0).
"""
import ctypes
import itertools
import math
import random

import numpy as np
import torch

import paper_2101_05031_gb300 as cs

DIRS = ((1, 0, 0), (0, 1, 0), (0, 0, 1), (1, 1, 0), (1, 0, 1), (0, 1, 1), (1, 1, 1))
LENGTH_DENSITY = 3.0 + 3.0 * math.sqrt(2.0) + math.sqrt(3.0)   # strut length per unit cell
GRADED_SPLIT = 0.165   # density at which the coarser of the two finest levels is split


def listed():
    return [
        # the smallest part (812 struts): launches and read-backs count
        dict(name="slice_cells", kind="slice", lattice="cells", n=4, spacing=5.0, nx=200, ny=200,
             pixel=0.1, dz=0.4, layers=50, ids=True, host=True),
        # one layer of a 429,039-strut part, as a streaming printer asks for it
        dict(name="slice_one_layer", kind="slice", lattice="grid", n=40, spacing=1.0, nx=2000,
             ny=2000, pixel=0.02, dz=0.2, layers=1, ids=False, host=True),
        # the whole of that part at 0.02 mm: supports of 26 pixels
        dict(name="slice_grid", kind="slice", lattice="grid", n=40, spacing=1.0, nx=2000, ny=2000,
             pixel=0.02, dz=0.2, layers=200, ids=False, host=False),
        # a graded part of 13 million fine struts at 0.05 mm: supports of 3.6 pixels
        dict(name="slice_graded", kind="slice", lattice="graded", box=100.0, level=7, nx=2000,
             ny=2000, pixel=0.05, dz=0.2, layers=500, ids=False, host=False),
        # upload and slicing of a 1.6-million-strut part from host arrays, odd sizes, edge ids
        dict(name="part_graded", kind="part", box=50.0, level=6, nx=1001, ny=997, pixel=0.05,
             dz=0.2, layers=247, ids=True),
        # the binary images of the largest part: 103 million struts, 4000^2 x 1000
        dict(name="mask_graded", kind="mask", lattice="graded", box=200.0, level=8, nx=4000,
             ny=4000, pixel=0.05, dz=0.2, layers=1000),
        # field and images of an odd-sized part, a few layers
        dict(name="field_grid", kind="field", lattice="grid", n=27, spacing=1.0, nx=1001, ny=787,
             pixel=0.035, dz=0.21, layers=13),
        # radius tuning of a million struts on 64^3 cells
        dict(name="tune_grid", kind="tune", n=53, spacing=1.0, dims=64, m=8),
        # twelve small parts as one graph
        dict(name="batch_grids", kind="batch", parts=12, most=200000, pixel=0.05, layers=100, mix=7),
        # post-processing of a part's contours for a laser: simplify, smooth, infill
        dict(name="finish_graded", kind="finish", box=50.0, level=6, nx=1000, ny=1000, pixel=0.05,
             dz=0.2, layers=250, hatch=0.1),
        # a lattice designed for voxel densities on a mesh of 93,750 tetrahedra
        dict(name="design_mesh", kind="design", cubes=25, edge=4.0, voxel=5.0),
        # a full-HD depth image of a 429,039-strut part
        dict(name="depth_grid", kind="depth", n=40, spacing=1.0, width=1920, height=1080),
    ]


def draw(rng):
    def between(lo, hi):   # spread over the logarithm
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(("slice", "slice", "slice", "part", "mask", "field", "tune", "batch",
                       "finish", "design", "depth"))
    if kind in ("slice", "mask", "field"):
        lattice = rng.choice(("cells", "grid", "grid", "graded", "graded"))
        c = dict(kind=kind, lattice=lattice)
        if lattice == "graded":
            level = rng.randint(5, 7)
            box = 100.0 / 2 ** (7 - level)
            px = rng.choice((0.04, 0.05, 0.06))
            c.update(box=box, level=level, pixel=px, nx=int(box / px) - rng.randint(0, 40),
                     ny=int(box / px) - rng.randint(0, 40), dz=0.2)
            full = int(box / 0.2)
        else:
            n = rng.randint(2, 6) if lattice == "cells" else between(8, 40)
            spacing = 5.0 if lattice == "cells" else 1.0
            px = rng.choice((0.05, 0.08, 0.1)) if lattice == "cells" else rng.choice((0.02, 0.03, 0.05))
            ext = n * spacing
            c.update(n=n, spacing=spacing, pixel=px, dz=rng.choice((0.15, 0.2, 0.4)),
                     nx=int(ext / px) - rng.randint(0, 37), ny=int(ext / px) - rng.randint(0, 37))
            full = min(200, int(ext / c["dz"]))
        c["layers"] = between(1, 40) if kind == "field" else between(1, full)
        if kind == "field":
            c["layers"] = min(c["layers"], full)
        if kind == "slice":
            c["ids"] = rng.random() < 0.5
            c["host"] = work(c)["bytes"] < 8e6
        return c
    if kind == "part":
        level = rng.randint(4, 6)
        box = 50.0 / 2 ** (6 - level)
        px = rng.choice((0.04, 0.05))
        return dict(kind="part", box=box, level=level, pixel=px, dz=0.2,
                    nx=int(box / px) - rng.randint(0, 9), ny=int(box / px) - rng.randint(0, 9),
                    layers=int(box / 0.2) - rng.randint(0, 9), ids=rng.random() < 0.5)
    if kind == "tune":
        n = between(9, 53)
        m = rng.choice((2, 4, 8, 8))
        return dict(kind="tune", n=n, spacing=1.0, m=m, dims=max(4, n * rng.randint(7, 10) // m))
    if kind == "batch":
        return dict(kind="batch", parts=rng.randint(2, 12), most=between(3000, 200000),
                    pixel=rng.choice((0.05, 0.06, 0.08)), layers=between(12, 100),
                    mix=rng.randint(0, 9999))
    if kind == "finish":
        level = rng.randint(4, 6)
        box = 50.0 / 2 ** (6 - level)
        px = rng.choice((0.04, 0.05))
        return dict(kind="finish", box=box, level=level, pixel=px, dz=0.2, hatch=0.1,
                    nx=int(box / px) - rng.randint(0, 9), ny=int(box / px) - rng.randint(0, 9),
                    layers=int(box / 0.2) - rng.randint(0, 9))
    if kind == "design":
        return dict(kind="design", cubes=between(3, 25), edge=4.0, voxel=rng.choice((4.5, 5.0, 6.0)))
    return dict(kind="depth", n=between(10, 40), spacing=1.0, width=between(320, 1920),
                height=between(240, 1080))


# --------------------------------------------------------------------------- inputs

def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _grid_lattice(dims, spacing, lo, hi, seed):
    """Jittered Freudenthal grid of dims nodes, jitter 0.2 spacing, radii U(lo, hi)."""
    g = _generator(seed)
    nx, ny, nz = dims
    ax = [torch.arange(k, device="cuda") for k in dims]
    ijk = torch.stack(torch.meshgrid(*ax, indexing="ij"), -1).reshape(-1, 3)
    jitter = torch.rand(ijk.shape, generator=g, device="cuda", dtype=torch.float64) * 0.4 - 0.2
    nodes = ((ijk + jitter) * spacing).float()
    ids = torch.arange(nx * ny * nz, device="cuda", dtype=torch.int32).reshape(nx, ny, nz)
    edges = torch.cat([torch.stack([ids[:nx - a, :ny - b, :nz - c].reshape(-1),
                                    ids[a:, b:, c:].reshape(-1)], 1) for a, b, c in DIRS])
    radius = torch.rand(edges.shape[0], generator=g, device="cuda") * (hi - lo) + lo
    return nodes, edges, radius


def _cell_lattice(n, cell, seed):
    """Cube edges and body diagonals of n^3 cells; radii U(0.4, 0.5), R = 0.75."""
    g = _generator(seed)
    ids = torch.arange((n + 1) ** 3, device="cuda").reshape(n + 1, n + 1, n + 1)
    mid = (n + 1) ** 3 + torch.arange(n ** 3, device="cuda").reshape(n, n, n)
    pairs = [(ids[:n + 1 - a, :n + 1 - b, :n + 1 - c], ids[a:, b:, c:]) for a, b, c in DIRS[:3]]
    pairs += [(mid, ids[a:n + a, b:n + b, c:n + c]) for a, b, c in itertools.product((0, 1), repeat=3)]
    edges = torch.cat([torch.stack([a.reshape(-1), b.reshape(-1)], 1) for a, b in pairs]).int()
    t = torch.arange(n + 1, device="cuda", dtype=torch.float64)
    corners = torch.cartesian_prod(t, t, t)
    centres = torch.cartesian_prod(t[:n], t[:n], t[:n]) + 0.5
    nodes = (torch.cat([corners, centres]) * cell).float()
    radius = torch.rand(edges.shape[0], generator=g, device="cuda") * 0.1 + 0.4
    return nodes, edges, radius


def _graded_r_ref(box, level):
    return box / 2 ** (level - 1) * math.sqrt(GRADED_SPLIT / (LENGTH_DENSITY * math.pi))


def _graded_lattice(box, level, seed):
    """Octree-graded Freudenthal lattice on [0, box]^3 with leaves of levels
    level - 1 and level: cubes are split where the target density (a wave in x
    and y whose phase comes from the seed) is above GRADED_SPLIT. Identical
    edges are kept once; the radius of a strut follows the target density."""
    g = _generator(seed)
    phase = torch.rand(2, generator=g, device="cuda", dtype=torch.float64) * 2 * math.pi
    k = 2 * math.pi / 50.0

    def density(x, y):
        return 0.1 + 0.3 * (0.5 + 0.5 * torch.sin(k * x + phase[0]) * torch.cos(k * y + phase[1]))

    r_ref = _graded_r_ref(box, level)
    n = 2 ** (level - 1)
    centre = (torch.arange(n, device="cuda", dtype=torch.float64) + 0.5) * (box / n)
    split = density(centre[:, None], centre[None, :]) > GRADED_SPLIT
    split = split[:, :, None].expand(n, n, n)
    leaves = ((n, ~split), (2 * n, split.repeat_interleave(2, 0).repeat_interleave(2, 1)
                            .repeat_interleave(2, 2)))
    nf = 2 * n + 1
    ends, used = [], torch.zeros(nf ** 3, dtype=torch.bool, device="cuda")
    for m, leaf in leaves:
        padded = torch.zeros((m + 2,) * 3, dtype=torch.bool, device="cuda")
        padded[1:-1, 1:-1, 1:-1] = leaf
        scale = 2 * n // m
        for d in DIRS:
            # an edge belongs to every leaf cube that touches it: the cube at
            # its lower node, and one step back along each axis it lies across
            has = torch.zeros((m + 1,) * 3, dtype=torch.bool, device="cuda")
            for back in itertools.product(*[(0, 1) if v == 0 else (0,) for v in d]):
                has |= padded[tuple(slice(1 - o, m + 2 - o) for o in back)]
            has = has[tuple(slice(0, m + 1 - v) for v in d)]
            i = torch.nonzero(has) * scale
            a = (i[:, 0] * nf + i[:, 1]) * nf + i[:, 2]
            b = a + ((d[0] * nf + d[1]) * nf + d[2]) * scale
            used[a] = True
            used[b] = True
            ends.append((box / m, a, b))
    fine = torch.nonzero(used).reshape(-1)
    ids = torch.full((nf ** 3,), -1, dtype=torch.int32, device="cuda")
    ids[fine] = torch.arange(fine.numel(), dtype=torch.int32, device="cuda")
    h = box / (nf - 1)
    nodes = torch.stack([fine // (nf * nf), fine // nf % nf, fine % nf], 1).double().mul_(h).float()
    edges, radius = [], []
    for cube, a, b in ends:
        x = ((a // (nf * nf)).double() + b // (nf * nf)) * (0.5 * h)
        y = ((a // nf % nf).double() + b // nf % nf) * (0.5 * h)
        r = torch.sqrt(density(x, y) / (LENGTH_DENSITY / cube ** 2 * math.pi))
        radius.append(r.clamp(0.25 * r_ref, r_ref).float())
        edges.append(torch.stack([ids[a], ids[b]], 1))
    return nodes, torch.cat(edges), torch.cat(radius)


def _lattice(case, seed):
    """nodes, edges, radius (on the GPU), R, and the extent of the box from 0."""
    which = case.get("lattice", "graded" if "box" in case else "grid")
    if which == "graded":
        return (*_graded_lattice(case["box"], case["level"], seed),
                1.5 * _graded_r_ref(case["box"], case["level"]), case["box"])
    if which == "cells":
        return (*_cell_lattice(case["n"], case["spacing"], seed), 0.75,
                case["n"] * case["spacing"])
    s = case["spacing"]
    return (*_grid_lattice((case["n"],) * 3, s, 0.15 * s, 0.35 * s, seed), 0.525 * s,
            (case["n"] - 1) * s)


def _window(case, extent):
    """Pixel window centred on the part, layers from its bottom."""
    px = case["pixel"]
    z = 0.5 * case["dz"]
    if case["layers"] * case["dz"] < 0.5 * extent:   # a few layers: from the middle up
        z += case["dz"] * int(0.5 * extent / case["dz"])
    return dict(x0=0.5 * (extent - case["nx"] * px), y0=0.5 * (extent - case["ny"] * px),
                nx=case["nx"], ny=case["ny"], pixel=px, z0=z, dz=case["dz"],
                n_layers=case["layers"])


def _batch_parts(case):
    """(node dims, spacing, largest radius) of every part: strut counts log-uniform
    up to `most`, boxes of 10 to 40 mm per axis."""
    r = random.Random(case["mix"])
    parts = []
    for _ in range(case["parts"]):
        struts = math.exp(r.uniform(math.log(1000), math.log(case["most"])))
        ext = [r.uniform(10.0, 40.0) for _ in range(3)]
        s = (7.0 * math.prod(ext) / struts) ** (1 / 3)
        parts.append((tuple(max(2, int(round(e / s)) + 1) for e in ext), s, min(0.5, 0.45 * s)))
    return parts


def _cells(case):
    n, s = case["n"], case["spacing"]
    return dict(origin=(-0.2 * s, -0.2 * s, -0.2 * s), h=(n - 0.6) * s / case["dims"],
                dims=(case["dims"],) * 3, m=case["m"], T=0.01)


def _tune_target(case, seed):
    g = _generator(seed + 77)
    return torch.rand((case["dims"],) * 3, generator=g, device="cuda") * 0.3 + 0.1


def _mesh(case, seed):
    """Jittered Kuhn mesh of a cube (six tetrahedra per cube) and a graded
    voxel target, host arrays."""
    c, h = case["cubes"], case["edge"]
    r = np.random.Generator(np.random.Philox(seed))
    ijk = np.stack(np.meshgrid(*[np.arange(c + 1)] * 3, indexing="ij"), -1).reshape(-1, 3)
    pos = ijk * h
    inner = ((ijk > 0) & (ijk < c)).all(1)
    pos[inner] += r.uniform(-0.1, 0.1, (int(inner.sum()), 3)) * h
    cube = np.stack(np.meshgrid(*[np.arange(c)] * 3, indexing="ij"), -1).reshape(-1, 3)
    tets = []
    for perm in itertools.permutations(range(3)):
        at, verts = cube.copy(), [cube]
        for ax in perm:
            at = at.copy()
            at[:, ax] += 1
            verts.append(at)
        tets.append(np.stack([(v[:, 0] * (c + 1) + v[:, 1]) * (c + 1) + v[:, 2] for v in verts], 1))
    tets = np.stack(tets, 1).reshape(-1, 4).astype(np.int32)
    v = case["voxel"]
    dims = max(1, math.ceil(c * h / v - 1e-9))
    at = v * (np.arange(dims) + 0.5)
    k, p = 2 * math.pi / 50.0, r.uniform(0, 2 * math.pi, 2)
    wave = 0.5 + 0.5 * np.sin(k * at[None, :] + p[0]) * np.cos(k * at[:, None] + p[1])
    target = (0.05 + 0.3 * wave)[None] * (1.0 + 0.2 * (np.arange(dims) + 0.5) / dims)[:, None, None]
    grid = dict(origin=(0.0, 0.0, 0.0), h=v, dims=(dims,) * 3, target=target.astype(np.float32))
    return pos.astype(np.float32), tets, grid


# --------------------------------------------------------------------------- a pass

def _room(layers, verts, ids, **where):
    """Buffers for contours of about `verts` vertices (loops have 4 or more)."""
    n = int((4 if verts < 2e7 else 1.6) * verts) + 20000
    room = dict(layers=torch.zeros(layers + 1, dtype=torch.int64, **where),
                loops=torch.zeros(n // 4 + 1, dtype=torch.int64, **where),
                xy=torch.zeros((n, 2), **where))
    if ids:
        room["edges"] = torch.zeros(n, dtype=torch.int32, **where)
    return room


def _room_for(state, verts, layers, ids):
    case = state["case"]
    if case["kind"] == "part":
        return _room(layers, verts, ids, pin_memory=True)
    if case.get("host"):
        return {k: t.numpy() for k, t in _room(layers, verts, ids).items()}
    return _room(layers, verts, ids, device="cuda")


def prepare(case, seed):
    kind = case["kind"]
    state = dict(case=case)
    if kind == "design":
        state["mesh"] = _mesh(case, seed)
        tets = state["mesh"][1].shape[0]
        state["room"] = {k: np.zeros((16 * tets + 500,) + w, t) for k, w, t in (
            ("nodes", (3,), np.float32), ("edges", (2,), np.int32), ("radius", (), np.float32),
            ("step3_ratio", (), np.float32), ("tets", (4,), np.int32), ("depth", (), np.int32),
            ("target", (), np.float64), ("rho_star", (), np.float32), ("tet_ratio", (), np.float32))}
        state["room"]["moves"] = np.zeros(100, np.int64)
        return state
    if kind == "batch":
        jobs = []
        for i, (dims, s, r) in enumerate(_batch_parts(case)):
            nodes, edges, radius = _grid_lattice(dims, s, min(0.1, 0.5 * r), r, seed * 64 + i)
            lat = cs.Lattice(nodes, edges, radius, R=0.75)
            ext = [(d - 1) * s for d in dims]
            nx, ny = (int(math.ceil((e + 2 * 0.75) / case["pixel"])) for e in ext[:2])
            dz = ext[2] / case["layers"]
            jobs.append((lat, dict(z0=0.5 * dz, dz=dz, n_layers=case["layers"], x0=-0.75, y0=-0.75,
                                   nx=nx, ny=ny, pixel=case["pixel"])))
        state["batch"] = cs.Batch(jobs)
        state["room"] = [_room(case["layers"], v, False, device="cuda")
                         for v in _batch_vertices(case)]
        return state
    nodes, edges, radius, R, extent = _lattice(case, seed)
    if kind == "part":
        state["arrays"] = tuple(t.cpu().pin_memory() for t in (nodes, edges, radius))
        state["R"], state["window"] = R, _window(case, extent)
        state["room"] = _room_for(state, _vertices(case), case["layers"], case["ids"])
        return state
    lat = state["lattice"] = cs.Lattice(nodes, edges, radius, R=R)
    if kind == "tune":
        state["nodes"], state["radius"] = nodes.requires_grad_(), radius.requires_grad_()
        state["target"] = _tune_target(case, seed)
        state["cells"] = _cells(case)
    elif kind == "depth":
        state["view"] = dict(eye=(1.6 * extent, -0.3 * extent, 1.2 * extent),
                             target=(0.5 * extent,) * 3, up=(0.0, 0.0, 1.0), fov_y=0.6,
                             width=case["width"], height=case["height"], step=R / 8, refine=20)
        state["out"] = torch.empty((case["height"], case["width"]), device="cuda")
    else:
        win = state["window"] = _window(case, extent)
        if kind == "finish":
            state["contours"] = lat.slice(**win, on_device=True, edge_ids=True)
            state["room"] = _room_for(state, _vertices(case), case["layers"], True)
            segments = state["room"]["xy"].shape[0] // 3
            state["room"].update(
                hatch_layers=torch.zeros(case["layers"] + 1, dtype=torch.int64, device="cuda"),
                hatch=torch.zeros((segments, 3), device="cuda"))
            state["lines"] = int(case["ny"] * case["pixel"] / case["hatch"])
        if kind == "slice":
            state["room"] = _room_for(state, _vertices(case), case["layers"], case["ids"])
        if kind in ("mask", "field"):
            state["mask"] = torch.empty((case["layers"], case["ny"], (case["nx"] + 31) // 32),
                                        dtype=torch.int32, device="cuda")
        if kind == "field":
            state["sigma"] = torch.empty((case["layers"], case["ny"], case["nx"]), device="cuda")
    return state


class _Device:
    """A library-owned device array, for torch."""

    def __init__(self, ptr, shape, kind):
        self.__cuda_array_interface__ = dict(shape=shape, typestr=kind, data=(ptr, False), version=2)


def _check(status):
    if status:
        raise RuntimeError(cs.load().csl_last_error().decode())


def _stream():
    return ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)


def _put(room, name, values):
    room[name][:len(values)] = values


def _take(contours, room):
    """Copies contours to the program's buffers (csl_contours_copy, or from the host arrays)."""
    if isinstance(contours, cs.ContourSet):
        _put(room, "layers", contours.layer_loop_off)
        _put(room, "loops", contours.loop_vert_off)
        _put(room, "xy", contours.xy)
        if "edges" in room:
            _put(room, "edges", contours.edge_id)
        return room
    if contours.n_verts > room["xy"].shape[0] or contours.n_loops >= room["loops"].shape[0]:
        raise RuntimeError("more contours than there is room for")
    at = [ctypes.c_void_p(room[k].data_ptr()) if k in room else None
          for k in ("layers", "loops", "xy", "edges")]
    _check(cs.load().csl_contours_copy(contours._ptr, *at, int(room["xy"].is_cuda), _stream()))
    return room


def run(state):
    case = state["case"]
    kind = case["kind"]
    room = state.get("room")
    if kind == "slice":
        return _take(state["lattice"].slice(**state["window"], edge_ids=case["ids"],
                                            on_device=not case["host"]), room)
    if kind == "part":
        lat = cs.Lattice(*state["arrays"], R=state["R"])
        return _take(lat.slice(**state["window"], edge_ids=case["ids"], on_device=True), room)
    if kind == "mask":
        state["lattice"].slice(**state["window"], contours=False, mask_out=state["mask"])
        return state["mask"]
    if kind == "field":
        state["lattice"].slice(**state["window"], contours=False, sigma_out=state["sigma"],
                               mask_out=state["mask"])
        return dict(sigma=state["sigma"], mask=state["mask"])
    if kind == "tune":
        vf = cs.VolumeFraction.apply(state["radius"], state["nodes"], state["lattice"],
                                     state["cells"])
        loss = (vf - state["target"]).square().sum()
        grad_radius, grad_nodes = torch.autograd.grad(loss, (state["radius"], state["nodes"]))
        return dict(vf=vf.detach(), grad_radius=grad_radius, grad_nodes=grad_nodes)
    if kind == "batch":
        state["batch"].run()
        for j in range(case["parts"]):
            out = ctypes.POINTER(cs._lib.Contours)()
            _check(cs.load().csl_batch_contours(state["batch"]._h, j, 1, ctypes.byref(out)))
            _take(cs.DeviceContours(out), room[j])
        return room
    if kind == "finish":
        px, win = case["pixel"], state["window"]
        c = state["contours"].simplify(case["nx"], case["ny"], 0.25 * px)
        c.smooth(win["x0"], win["y0"], px, case["nx"], case["ny"], lam=0.5, margin=0.05, iterations=4)
        _take(c, room)
        lib, out = cs.load(), ctypes.POINTER(cs._lib.Hatches)()
        _check(lib.csl_hatch_layers(c._ptr, win["y0"] + 0.5 * case["hatch"], case["hatch"],
                                    state["lines"], 1, _stream(), ctypes.byref(out)))
        h = out.contents
        _put(room, "hatch_layers", torch.as_tensor(
            _Device(h.layer_seg_off, (h.n_layers + 1,), "<i8"), device="cuda"))
        _put(room, "hatch", torch.as_tensor(_Device(h.seg, (h.n_segments, 3), "<f4"), device="cuda"))
        lib.csl_hatches_free(out)
        return room
    if kind == "design":
        nodes, tets, grid = state["mesh"]
        moved = cs.support_optimize(nodes, tets)
        made = cs.density_match(moved["nodes"], tets, grid, r_min=0.1)
        for k in room:
            if k != "moves":
                _put(room, k, made[k])
        _put(room, "moves", moved["moves_per_round"])
        return dict(room, moved=moved["nodes"], gamma=moved["gamma_after"], psi=moved["psi_after"],
                    voxel_ratio=made["voxel_ratio"])
    if kind == "depth":
        return state["lattice"].render_depth(**state["view"], out=state["out"])
    raise ValueError(kind)


# --------------------------------------------------------------------------- work

def _size(case):
    """(nodes, struts, total strut length, mean radius, R, extent) of a case's lattice."""
    which = case.get("lattice", "graded" if "box" in case else "grid")
    if which == "graded":
        box, level = case["box"], case["level"]
        fine = 2 ** level
        share = 0.75   # of the volume that the target density splits
        cubes = fine ** 3 * (share + (1 - share) / 8)
        length = box ** 3 * LENGTH_DENSITY * (share * (fine / box) ** 2
                                              + (1 - share) * (fine / 2 / box) ** 2)
        r = _graded_r_ref(box, level)
        return 1.05 * cubes, 7.2 * cubes, length, 0.75 * r, 1.5 * r, box
    if which == "cells":
        n, s = case["n"], case["spacing"]
        struts = 3 * n * (n + 1) ** 2 + 8 * n ** 3
        length = (3 * n * (n + 1) ** 2 + 4 * math.sqrt(3.0) * n ** 3) * s
        return (n + 1) ** 3 + n ** 3, struts, length, 0.45, 0.75, n * s
    n, s = case["n"], case["spacing"]
    struts = sum((n - a) * (n - b) * (n - c) for a, b, c in DIRS)
    return n ** 3, struts, 1.03 * LENGTH_DENSITY / 7 * struts * s, 0.25 * s, 0.525 * s, (n - 1) * s


def _share(case, extent):
    """The share of the part inside the window."""
    return min(1.0, case["nx"] * case["pixel"] / extent) * \
        min(1.0, case["ny"] * case["pixel"] / extent) * min(1.0, case["layers"] * case["dz"] / extent)


def _vertices(case):
    """About how many contour vertices a case has: one per pixel of perimeter and axis."""
    _, _, length, r, _, extent = _size(case)
    return 0.6 * _share(case, extent) * 2 * math.pi * r * length / case["pixel"] / case["dz"]


def _batch_vertices(case):
    out = []
    for dims, s, r in _batch_parts(case):
        dz = (dims[2] - 1) * s / case["layers"]
        area = 2 * math.pi * 0.6 * r * LENGTH_DENSITY * s * math.prod(dims)
        out.append(0.6 * area / case["pixel"] / dz)
    return out


def work(case):
    """Bytes: inputs read once and outputs written once. Flops: 36 for each nonzero
    (sample, strut) term of the field; its gradients 124 more."""
    kind = case["kind"]
    if kind == "design":
        tets = 6 * case["cubes"] ** 3
        leaves = 3.8 * tets
        samples = 8 ** 3 * leaves
        return dict(bytes=16.0 * tets + 12.0 * (case["cubes"] + 1) ** 3 + 60.0 * leaves,
                    flops=samples * (6 * 36 + 26 * 8))
    if kind == "batch":
        total = dict(bytes=0.0, flops=0.0)
        for (dims, s, r), verts in zip(_batch_parts(case), _batch_vertices(case)):
            n = math.prod(dims)
            length = LENGTH_DENSITY * s * n
            cell = case["pixel"] ** 2 * (dims[2] - 1) * s / case["layers"]
            total["bytes"] += (12 + 12 * 7) * n + 8 * verts
            total["flops"] += 36 * length * math.pi * 0.75 ** 2 / cell
        return total
    nodes, struts, length, r, R, extent = _size(case)
    read = 12.0 * nodes + 12.0 * struts
    if kind == "tune":
        px = (case["n"] - 0.6) * case["spacing"] / case["dims"] / case["m"]
        terms = length * math.pi * R ** 2 / px ** 3
        return dict(bytes=2 * read + 8.0 * case["dims"] ** 3,
                    flops=terms * (2 * 36 + 0.1 * 124))
    if kind == "depth":
        rays = float(case["width"]) * case["height"]
        return dict(bytes=read + 4 * rays, flops=rays * 40 * 8 * 36)
    share, verts = _share(case, extent), _vertices(case)
    pixels = float(case["nx"]) * case["ny"] * case["layers"]
    terms = share * length * math.pi * R ** 2 / (case["pixel"] ** 2 * case["dz"])
    if kind == "finish":
        return dict(bytes=12 * verts + 12 * 0.6 * verts + 0.13 * 12 * verts, flops=60 * verts)
    out = {"mask": pixels / 8, "field": pixels * 4.125}.get(kind, verts * (12 if case.get("ids") else 8))
    return dict(bytes=share * read + out, flops=36 * terms)


# --------------------------------------------------------------------------- 64 bits

def _terms64(a, b, w, R, x, y, z, budget=1 << 25):
    """Yields (struts, rows, columns, strut rows of the list) of the samples
    (x[i], y[j], z) within R of each strut, in pieces of bounded size."""
    near = torch.nonzero((torch.minimum(a[:, 2], b[:, 2]) <= z + R)
                         & (torch.maximum(a[:, 2], b[:, 2]) >= z - R)).reshape(-1)
    if near.numel() == 0:
        return
    A, D = a[near], b[near] - a[near]
    dz = torch.where(D[:, 2] == 0, torch.ones_like(D[:, 2]), D[:, 2])
    flat = D[:, 2] == 0
    t = torch.stack([(z - R - A[:, 2]) / dz, (z + R - A[:, 2]) / dz], 1).clamp(0, 1)
    t = torch.where(flat[:, None], torch.tensor([0.0, 1.0], device="cuda", dtype=t.dtype), t)
    ends = A[:, None, :2] + t[:, :, None] * D[:, None, :2]
    lo, hi = ends.amin(1) - R, ends.amax(1) + R
    px, py = float(x[1] - x[0]), float(y[1] - y[0])
    first = torch.stack([((lo[:, 0] - x[0]) / px).ceil(), ((lo[:, 1] - y[0]) / py).ceil()], 1).long()
    last = torch.stack([((hi[:, 0] - x[0]) / px).floor(), ((hi[:, 1] - y[0]) / py).floor()], 1).long()
    top = torch.tensor([x.numel() - 1, y.numel() - 1], device="cuda")
    first, last = torch.maximum(first, torch.zeros_like(first)), torch.minimum(last, top)
    keep = (first <= last).all(1)
    near, first, last = near[keep], first[keep], last[keep]
    if near.numel() == 0:
        return
    wide, high = (int(v) for v in (last - first + 1).amax(0))
    di = torch.arange(wide, device="cuda")
    dj = torch.arange(high, device="cuda")
    step = max(1, budget // (wide * high))
    for s in range(0, near.numel(), step):
        k = near[s:s + step]
        i, j = first[s:s + step, 0, None] + di, first[s:s + step, 1, None] + dj
        X = x[i.clamp(max=x.numel() - 1)] - a[k, 0, None]
        Y = y[j.clamp(max=y.numel() - 1)] - a[k, 1, None]
        Z = (z - a[k, 2])[:, None, None]
        u = b[k] - a[k]
        u = u / u.norm(dim=1, keepdim=True).clamp(min=1e-300)
        along = X[:, None, :] * u[:, 0, None, None] + Y[:, :, None] * u[:, 1, None, None] \
            + Z * u[:, 2, None, None]
        gap = (X * X)[:, None, :] + (Y * Y)[:, :, None] + Z * Z - along * along
        hit = (gap < R * R) & (i <= last[s:s + step, 0, None])[:, None, :] \
            & (j <= last[s:s + step, 1, None])[:, :, None]
        q, jj, ii = torch.nonzero(hit, as_tuple=True)
        yield k, j[q, jj], i[q, ii], q


def _integral64(a, b, x, y, z, R):
    """The quartic kernel's integral along each segment a-b at points (x, y, z)."""
    d = b - a
    length = d.norm(dim=1)
    u = d / length[:, None]
    p = torch.stack([x, y, z], 1) - a
    t0 = (p * u).sum(1)
    h2 = R * R - ((p - t0[:, None] * u) ** 2).sum(1)
    on = h2 > 0
    h2 = torch.where(on, h2, torch.ones_like(h2))
    w = h2.sqrt()
    lo, hi = torch.maximum(-t0, -w), torch.minimum(length - t0, w)
    on = on & (hi > lo)

    def prim(t):
        return t * (h2 * h2 - t * t * (2.0 / 3.0 * h2 - 0.2 * t * t))

    return torch.where(on, prim(hi) - prim(lo), torch.zeros_like(h2)) / R ** 4


def _weight64(radius, R):
    return 15.0 * R ** 4 / (16.0 * (R * R - radius * radius) ** 2.5)


def _plane64(a, b, w, R, x, y, z):
    plane = torch.zeros(y.numel() * x.numel(), device="cuda", dtype=torch.float64)
    for k, j, i, q in _terms64(a, b, w, R, x, y, z):
        e = k[q]
        v = w[e] * _integral64(a[e], b[e], x[i], y[j], torch.full_like(x[i], z), R)
        plane.index_add_(0, j * x.numel() + i, v)
    return plane.reshape(y.numel(), x.numel())


def exact(case, seed):
    if case["kind"] not in ("field", "tune"):
        return None   # contours, images and meshes: their topology is decided by rounding
    nodes, edges, radius, R, extent = _lattice(case, seed)
    if case["kind"] == "field":
        a, b = nodes[edges[:, 0]].double(), nodes[edges[:, 1]].double()
        w, win = _weight64(radius.double(), R), _window(case, extent)
        if work(case)["flops"] > 36e10:   # takes too long
            return None
        x = win["x0"] + (torch.arange(win["nx"], device="cuda").double() + 0.5) * win["pixel"]
        y = win["y0"] + (torch.arange(win["ny"], device="cuda").double() + 0.5) * win["pixel"]
        sigma = torch.stack([_plane64(a, b, w, R, x, y, win["z0"] + k * win["dz"])
                             for k in range(win["n_layers"])])
        return dict(sigma=sigma, mask=None)
    cells = _cells(case)
    dims, m, T = case["dims"], case["m"], cells["T"]
    px = cells["h"] / m
    at = cells["origin"][0] + (torch.arange(dims * m, device="cuda").double() + 0.5) * px
    target = _tune_target(case, seed).double()
    nodes, radius = nodes.double().requires_grad_(), radius.double().requires_grad_()
    a, b = (nodes.detach()[edges[:, c]] for c in (0, 1))
    w = _weight64(radius.detach(), R)
    vf = []
    for cz in range(dims):
        soft = sum(torch.sigmoid((_plane64(a, b, w, R, at, at, float(at[cz * m + k])) - 1.0) / T)
                   for k in range(m))
        vf.append(soft.reshape(dims, m, dims, m).sum((1, 3)) / m ** 3)
    vf = torch.stack(vf)
    slope = 2 * (vf - target) / m ** 3
    grad_radius, grad_nodes = torch.zeros_like(radius), torch.zeros_like(nodes)
    for l in range(dims * m):
        z = float(at[l])
        s = torch.sigmoid((_plane64(a, b, w, R, at, at, z) - 1.0) / T)
        alpha = (slope[l // m].repeat_interleave(m, 0).repeat_interleave(m, 1) * s * (1 - s) / T)
        for k, j, i, q in _terms64(a, b, w, R, at, at, z):
            live = alpha[j, i] != 0
            j, i, e = j[live], i[live], k[q[live]]
            if e.numel() == 0:
                continue
            A, B, r = (t[e].detach().requires_grad_() for t in (a, b, radius))
            f = _weight64(r, R) * _integral64(A, B, at[i], at[j], torch.full_like(at[i], z), R)
            ga, gb, gr = torch.autograd.grad(f, (A, B, r), alpha[j, i])
            grad_radius.index_add_(0, e, gr)
            grad_nodes.index_add_(0, edges[e, 0].long(), ga)
            grad_nodes.index_add_(0, edges[e, 1].long(), gb)
    return dict(vf=vf, grad_radius=grad_radius.detach(), grad_nodes=grad_nodes.detach())
