"""What is timed when this library is measured: ghost fills, their adjoints,
the fill fused with its stencil and the box packing of the exchange, each
through the public entry points of :mod:`paper_2605_14780_gb300.bc` with the
plan's default options.

A case names a grid (``sphere``: six equiangular gnomonic panels; ``blocks``:
uneven 2-D blocks with one drawn boundary condition per edge; ``box``: 3-D
blocks; ``nodes``: node-centred blocks that share their edges), its sizes,
the memory layout of the levels (``outer``: ``[level][k][j][i]``, ``inner``:
``[k][j][i][level]``), the dtype and the pass.  Field values are made on the
GPU from the seed; block shapes and boundary types are part of the case.

:func:`exact` restates the operator in FP64 from its definition: a list of
links, each "these ghost cells are weighted sums of those data cells".
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_2605_14780_gb300 import bc

HALO_TYPES = ("halo", "circular", "symmetric", "zero", "csr")
STENCIL_27 = bc.box_stencil(3, 1)
COEFFS_27 = np.array([26.0 if not o.any() else -1.0 for o in STENCIL_27])


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------
def listed():
    return [
        # one scalar on a tiny sphere: the latency of a call (two kernel
        # families of a few warps each)
        dict(name="sphere32_f64_fwd", grid="sphere", n=32, h=2, p=4, quad=0, levels=1,
             fields="scalar", dtype="f64", layout="outer", op="forward"),
        # faces of one 128^3 block, x periodic: the ghost fill between two
        # operator applications of an HPCG-like solver
        dict(name="box128_f64_fwd", grid="box", n0=128, n1=128, n2=128, nblocks=1, faces="P",
             dtype="f64", op="forward"),
        # many uneven blocks (multi-block model, halo / periodic / mirror /
        # zero / user CSR edges) in one call, levels contiguous
        dict(name="blocks512_inner_fwd", grid="blocks", nblocks=512, lo=16, hi=256, levels=64,
             h=2, mix=4, dtype="f32", layout="inner", op="forward"),
        # the same blocks with one plane per level
        dict(name="blocks512_outer_fwd", grid="blocks", nblocks=512, lo=16, hi=256, levels=64,
             h=2, mix=4, dtype="f32", layout="outer", op="forward"),
        # its gradient: cotangents of the ghosts added back into the data
        dict(name="blocks512_inner_adj", grid="blocks", nblocks=512, lo=16, hi=256, levels=64,
             h=2, mix=4, dtype="f32", layout="inner", op="adjoint"),
        # shallow-water sphere, (h, u, v) x 32 levels: 6-point edge
        # interpolation and rotated winds, once per time step
        dict(name="sphere384_f32_fwd", grid="sphere", n=384, h=3, p=6, quad=0, levels=32,
             fields="huv", dtype="f32", layout="outer", op="forward"),
        # adjoint model of a finer sphere
        dict(name="sphere768_f32_adj", grid="sphere", n=768, h=3, p=6, quad=0, levels=32,
             fields="huv", dtype="f32", layout="outer", op="adjoint"),
        # cell averages: reconstruction x quadrature rows (16 / 32 entries)
        dict(name="sphere384_quad_fwd", grid="sphere", n=384, h=3, p=4, quad=2, levels=32,
             fields="huv", dtype="f32", layout="outer", op="forward"),
        # an odd FP64 sphere with contiguous levels: forward and adjoint of
        # one assimilation step
        dict(name="sphere91_f64_both", grid="sphere", n=91, h=3, p=6, quad=0, levels=37,
             fields="huv", dtype="f64", layout="inner", op="both"),
        # node-centred blocks: halo copies and averaging of shared nodes
        dict(name="nodes8x8_f32_fwd", grid="nodes", bx=8, by=8, n=129, h=3, comps=3, levels=32,
             dtype="f32", layout="outer", op="forward"),
        # the fill fused with the 27-point operator that reads it
        dict(name="box16x128_f64_stencil", grid="box", n0=128, n1=128, n2=128, nblocks=16,
             faces="P", dtype="f64", op="stencil"),
        # edge strips of a quarter of the blocks packed for other ranks
        dict(name="blocks512_inner_pack", grid="blocks", nblocks=512, lo=16, hi=256, levels=64,
             h=2, mix=4, dtype="f32", layout="inner", op="pack"),
    ]


def draw(rng):
    def logint(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    grid = rng.choice(["sphere", "sphere", "sphere", "blocks", "blocks", "box", "nodes"])
    dtype = rng.choice(["f32", "f32", "f64"])
    layout = rng.choice(["outer", "inner"])
    if grid == "sphere":
        quad = rng.choice([0, 0, 2])
        n = logint(24, 300 if quad else 640)
        return dict(grid=grid, n=n, h=rng.choice([2, 3]), p=4 if quad else rng.choice([4, 6]),
                    quad=quad, levels=logint(1, 40), fields=rng.choice(["scalar", "huv", "huv"]),
                    dtype=dtype, layout=layout,
                    op=rng.choice(["forward", "forward", "adjoint", "both"]))
    if grid == "blocks":
        return dict(grid=grid, nblocks=logint(8, 512), lo=16, hi=logint(32, 256),
                    levels=logint(2, 64), h=rng.choice([1, 2, 3]), mix=rng.randrange(1000),
                    dtype=dtype, layout=layout,
                    op=rng.choice(["forward", "forward", "adjoint", "pack"]))
    if grid == "box":
        return dict(grid=grid, n0=logint(16, 160), n1=logint(16, 160), n2=logint(16, 160),
                    nblocks=logint(1, 8), faces=rng.choice("ZPS"), dtype=dtype,
                    op=rng.choice(["forward", "stencil"]))
    return dict(grid=grid, bx=rng.randint(2, 8), by=rng.randint(2, 8), n=logint(9, 129),
                h=rng.choice([2, 3]), comps=rng.randint(1, 3), levels=logint(1, 32), dtype=dtype,
                layout=layout, op=rng.choice(["forward", "forward", "adjoint"]))


# ---------------------------------------------------------------------------
# grids: blocks and boundary descriptions (the vocabulary of the package's
# specs module)
# ---------------------------------------------------------------------------
def _block(n, h, levels, comps):
    return {"n": tuple(int(v) for v in n), "h": tuple(int(v) for v in h),
            "nlevels": int(levels), "ncomp": int(comps)}


def _grid(case):
    return {"sphere": _sphere, "blocks": _blocks, "box": _box, "nodes": _nodes}[case["grid"]](case)


def _sphere(case):
    n, h = case["n"], case["h"]
    huv = case["fields"] == "huv"
    scal, pair = [0], [1, 2] if huv else None
    blocks = [_block((n, n, 1), (h, h, 0), case["levels"], 3 if huv else 1) for _ in range(6)]
    edges = {"kind": "cubed_sphere_edges", "panels": list(range(6)), "N": n, "h": h,
             "p": case["p"], "scalar_comps": scal, "vector_pair": pair}
    if case["quad"]:
        edges["quad"] = case["quad"]
    bcs = [edges]
    for panel in range(6):
        for ci, cj in ((0, 0), (n - 1, 0), (0, n - 1), (n - 1, n - 1)):
            bcs.append(_corner(n, h, panel, ci, cj, scal, pair))
    return blocks, bcs


def _corner(n, h, panel, ci, cj, scal, pair):
    """The h x h ghosts at one panel corner: a scalar is the mean of the
    three cells that meet at the cube vertex, a vector component a copy of
    the panel's own corner cell."""
    own = np.sign(_cell_point(n, panel, ci, cj))
    meet = [(q, i, j) for q in range(6) for i in (0, n - 1) for j in (0, n - 1)
            if (np.sign(_cell_point(n, q, i, j)) == own).all()]
    lo = (-h if ci == 0 else n, -h if cj == 0 else n, 0)
    cells = h * h
    ptr, blk, comp, ijk, val = [0], [], [], [], []
    for c in scal + (pair or []):
        src = meet if c in scal else [(panel, ci, cj)]
        for _ in range(cells):
            for q, i, j in src:
                blk.append(q)
                comp.append(c)
                ijk.append((i, j, 0))
                val.append(1.0 / len(src))
            ptr.append(len(val))
    return {"kind": "csr", "block": panel, "lo": lo, "hi": (lo[0] + h, lo[1] + h, 1),
            "comps": scal + (pair or []), "row_ptr": np.array(ptr, np.int64),
            "col_block": np.array(blk, np.int32), "col_comp": np.array(comp, np.int32),
            "col_ijk": np.array(ijk, np.int32), "val": np.array(val), "rhs": None}


def _blocks(case):
    """2-D blocks with log-uniform sides and uniform level counts; every edge
    draws a boundary type (a halo edge needs a partner of the same length
    and level count), corners are zero."""
    rng = random.Random(case["mix"])
    nrng = np.random.default_rng(case["mix"])
    h, lo, hi = case["h"], case["lo"], case["hi"]
    blocks = []
    for _ in range(case["nblocks"]):
        nx, ny = (min(hi, int(math.exp(rng.uniform(math.log(lo), math.log(hi + 1)))))
                  for _ in range(2))
        blocks.append(_block((nx, ny, 1), (h, h, 0), rng.randint(1, case["levels"]), 1))
    edges = {}
    for b, blk in enumerate(blocks):
        for axis in (0, 1):
            for side in (0, 1):
                edges.setdefault((blk["n"][1 - axis], blk["nlevels"]), []).append((b, axis, side))
    bcs = []
    for b, blk in enumerate(blocks):
        faces = []
        for axis in (0, 1):
            for side in (0, 1):
                length, depth = blk["n"][1 - axis], min(8, blk["n"][axis])
                partners = [e for e in edges[(length, blk["nlevels"])] if e != (b, axis, side)]
                t = rng.choice(HALO_TYPES if partners else HALO_TYPES[1:])
                face = {"axis": axis, "side": side, "type": t}
                if t == "halo":
                    sb, sa, ss = rng.choice(partners)
                    face.update(src_block=sb, src_axis=sa, src_side=ss, flip=rng.randrange(2))
                elif t == "csr":  # 2..8 of the first 8 layers, weights summing to one
                    nnz = np.minimum(nrng.integers(2, 9, size=(h, length)), depth)
                    on = np.arange(depth) < nnz[..., None]
                    order = np.argsort(nrng.random((h, length, depth)), axis=-1)
                    layers = np.sort(np.where(on, order, depth), axis=-1) * on
                    w = (1.0 - nrng.random((h, length, depth))) * on
                    face.update(nnz=nnz, layers=layers, weights=w / w.sum(-1, keepdims=True))
                faces.append(face)
        bcs.append({"kind": "faces", "block": b, "corners": "zero", "faces": faces})
    return blocks, bcs


def _box(case):
    blocks = [_block((case["n0"], case["n1"], case["n2"]), (1, 1, 1), 1, 1)
              for _ in range(case["nblocks"])]
    kinds = {"Z": {}, "P": {0: "circular"}, "S": {1: "symmetric"}}[case["faces"]]
    return blocks, [{"kind": "faces", "block": b, "corners": "product",
                     "faces": [{"axis": a, "side": s, "type": kinds.get(a, "zero")}
                               for a in range(3) for s in (0, 1)]}
                    for b in range(case["nblocks"])]


def _copies(case, a, b, i, j):
    """Every stored copy (block, i, j) of node (i, j) of block (a, b)."""
    n, bx, by = case["n"], case["bx"], case["by"]

    def along(k, blk, count):
        out = [(blk, k)]
        if k == 0 and blk > 0:
            out.append((blk - 1, n - 1))
        if k == n - 1 and blk < count - 1:
            out.append((blk + 1, 0))
        return out
    return sorted((jb * bx + ib, ii, jj) for ib, ii in along(i, a, bx)
                  for jb, jj in along(j, b, by))


def _nodes(case):
    n, h, bx, by = case["n"], case["h"], case["bx"], case["by"]
    comps = list(range(case["comps"]))
    blocks = [_block((n, n, 1), (h, h, 0), case["levels"], case["comps"])
              for _ in range(bx * by)]
    bcs = []
    for b in range(by):
        for a in range(bx):
            k = b * bx + a
            cols = [i for i, on in ((0, a > 0), (n - 1, a < bx - 1)) if on]
            boxes = [((i, 0), (i + 1, n)) for i in cols]
            i0, i1 = (1 if 0 in cols else 0), (n - 1 if n - 1 in cols else n)
            boxes += [((i0, j), (i1, j + 1)) for j, on in ((0, b > 0), (n - 1, b < by - 1)) if on]
            for lo, hi in boxes:
                groups = [_copies(case, a, b, i, j) for j in range(lo[1], hi[1])
                          for i in range(lo[0], hi[0])]
                sizes = np.array([len(g) for g in groups])
                ijk = np.array([(i, j, 0) for g in groups for _, i, j in g], np.int32)
                blk = np.array([q for g in groups for q, _, _ in g], np.int32)
                m = len(comps)
                bcs.append({"kind": "sync", "block": k, "lo": lo + (0,), "hi": hi + (1,),
                            "comps": comps,
                            "row_ptr": np.concatenate([[0], np.cumsum(np.tile(sizes, m))]),
                            "col_block": np.tile(blk, m),
                            "col_comp": np.repeat(np.array(comps, np.int32), len(blk)),
                            "col_ijk": np.tile(ijk, (m, 1)),
                            "val": np.tile(np.repeat(1.0 / sizes, sizes), m), "rhs": None})
            for axis in (0, 1):
                for side in (0, 1):
                    lo, hi = [0, 0, 0], [n, n, 1]
                    lo[axis], hi[axis] = (n, n + h) if side else (-h, 0)
                    na, nb = (a + (1 if side else -1), b) if axis == 0 else (a, b + (1 if side else -1))
                    d = {"block": k, "lo": tuple(lo), "hi": tuple(hi), "comps": comps}
                    if 0 <= na < bx and 0 <= nb < by:  # skips the shared line
                        off = [0, 0, 0]
                        off[axis] = 1 - n if side else n - 1
                        bcs.append(dict(d, kind="map", src_block=nb * bx + na, perm=(0, 1, 2),
                                        sign=(1, 1, 1), offset=tuple(off)))
                    else:
                        bcs.append(dict(d, kind="zero"))
            for x in ((-h, 0), (n, n + h)):
                for y in ((-h, 0), (n, n + h)):
                    bcs.append({"kind": "zero", "block": k, "lo": (x[0], y[0], 0),
                                "hi": (x[1], y[1], 1), "comps": comps})
    return blocks, bcs


# ---------------------------------------------------------------------------
# memory: all blocks of a field set in one buffer
# ---------------------------------------------------------------------------
def _full(blk):
    return [blk["n"][d] + 2 * blk["h"][d] for d in range(3)]


class _Layout:
    """Block b, component c, level l, cell q (axis 0 fastest over the full
    region) is element ``first[b] + c * comp[b] + l * lev[b] + q * cell[b]``."""

    def __init__(self, blocks, layout):
        self.blocks, self.inner = blocks, layout == "inner"
        self.first, self.size = [], 0
        for blk in blocks:
            self.first.append(self.size)
            values = blk["ncomp"] * blk["nlevels"] * math.prod(_full(blk))
            self.size += -(-values // 128) * 128  # blocks start on 512 bytes or more
        self.cells = [math.prod(_full(blk)) for blk in blocks]
        self.comp = [c * blk["nlevels"] for c, blk in zip(self.cells, blocks)]
        self.cell = [blk["nlevels"] if self.inner else 1 for blk in blocks]
        self.lev = [1 if self.inner else c for c in self.cells]

    def views(self, buf):
        """Per block a tensor indexed (component, level, k, j, i)."""
        out = []
        for b, blk in enumerate(self.blocks):
            f = _full(blk)
            s = self.cell[b]
            out.append(buf.as_strided((blk["ncomp"], blk["nlevels"], f[2], f[1], f[0]),
                                      (self.comp[b], self.lev[b], s * f[0] * f[1], s * f[0], s),
                                      self.first[b]))
        return out

    def cell_index(self, b, ijk):
        """Cell numbers of data coordinates ``ijk`` (..., 3)."""
        blk = self.blocks[b]
        f, h = _full(blk), blk["h"]
        ijk = np.asarray(ijk, np.int64)
        return ((ijk[..., 2] + h[2]) * f[1] + ijk[..., 1] + h[1]) * f[0] + ijk[..., 0] + h[0]

    def where(self, b, c, cells, device):
        """Elements (cell, level) of cells of one component."""
        q = torch.as_tensor(np.asarray(cells), device=device).reshape(-1, 1)
        lev = torch.arange(self.blocks[b]["nlevels"], device=device)
        return self.first[b] + c * self.comp[b] + q * self.cell[b] + lev * self.lev[b]


def _layout(case):
    blocks, _ = _grid(case)
    return _Layout(blocks, case.get("layout", "outer"))


def _data(view, blk):
    n, h = blk["n"], blk["h"]
    return view[:, :, h[2]:h[2] + n[2], h[1]:h[1] + n[1], h[0]:h[0] + n[0]]


def _fields(case, lay, seed, dev, ghosts):
    """Field values: data as the workload has it, ghosts NaN (never read
    before they are filled) or, for cotangents, uniform like the data."""
    dt = torch.float32 if case["dtype"] == "f32" else torch.float64
    gen = torch.Generator(device=dev).manual_seed(seed)
    if ghosts:
        return torch.rand(lay.size, generator=gen, device=dev, dtype=dt) * 2 - 1
    buf = torch.full((lay.size,), math.nan, device=dev, dtype=dt)
    for b, (view, blk) in enumerate(zip(lay.views(buf), lay.blocks)):
        d = _data(view, blk)
        if case["grid"] == "sphere" and case["fields"] == "huv":
            _weather(d, b, case["n"], seed, dev)
        else:
            low = 0.0 if case["grid"] == "box" else -1.0
            d.copy_(torch.rand(d.shape, generator=gen, device=dev, dtype=dt) * (1 - low) + low)
    last = lay.first[-1] + lay.blocks[-1]["ncomp"] * lay.comp[-1]
    for start, stop in zip([f + b["ncomp"] * c for f, b, c in
                            zip(lay.first, lay.blocks, lay.comp)], lay.first[1:] + [lay.size]):
        buf[start:stop] = 0  # padding between blocks
    buf[last:] = 0
    return buf


def _weather(d, panel, n, seed, dev):
    """Smooth height (1e4 +- 100 m) and covariant components of a rigid
    rotation (50 m/s) about an axis of its own per level."""
    rng = np.random.default_rng(seed)
    dirs = rng.normal(size=(6, 3))
    axes = rng.normal(size=(d.shape[1], 3))
    axes /= np.linalg.norm(axes, axis=1, keepdims=True)
    scale = rng.uniform(0.5, 1.0, size=d.shape[1])
    j, i = np.meshgrid(np.arange(n), np.arange(n), indexing="ij")
    a, b = _angle(n, i.ravel()), _angle(n, j.ravel())
    r, ea, eb = _basis(panel, a, b)
    height = np.sin(r @ dirs.T * 2).sum(1) / 6
    f64 = dict(dtype=torch.float64, device=dev)
    t = {k: torch.as_tensor(v, **f64) for k, v in
         (("r", r), ("ea", ea), ("eb", eb), ("h", height), ("ax", axes), ("s", scale))}
    wind = lambda e: 50.0 * t["ax"] @ torch.linalg.cross(t["r"], e).T  # noqa: E731
    shape = d.shape[1:]
    d[0].copy_((1e4 + 100.0 * t["s"][:, None] * t["h"]).reshape(shape))
    d[1].copy_(wind(t["ea"]).reshape(shape))
    d[2].copy_(wind(t["eb"]).reshape(shape))


def _strips(case, blocks):
    """The boxes other ranks ask for: the first ``h`` layers behind every
    edge of each fourth block."""
    h = case["h"]
    out = []
    for b in range(0, len(blocks), 4):
        n = blocks[b]["n"]
        for axis in (0, 1):
            for side in (0, 1):
                lo, hi = [0, 0, 0], list(n)
                lo[axis], hi[axis] = (n[axis] - h, n[axis]) if side else (0, h)
                out.append((b, tuple(lo), tuple(hi)))
    return out


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def prepare(case, seed):
    blocks, bcs = _grid(case)
    lay = _Layout(blocks, case.get("layout", "outer"))
    op = case["op"]
    buf = _fields(case, lay, seed, "cuda", ghosts=op == "adjoint")
    views = lay.views(buf)
    state = {"op": op, "fields": buf, "table": bc.slot_table(views)}
    if op == "pack":
        state["pack"] = bc.Pack(bc.block_descriptors(views, blocks), _strips(case, blocks),
                                case["dtype"])
        state["buffer"] = torch.empty(state["pack"].size, dtype=buf.dtype, device="cuda")
        return state
    w = {"blocks": blocks, "bcs": bcs, "dtype": case["dtype"]}
    state["plan"] = bc.plan_for_workload(w, views,
                                         {"stencil_fusion": 1} if op == "stencil" else None)
    if op == "both":
        state["cotangent"] = _fields(case, lay, seed + 1_000_003, "cuda", ghosts=True)
        state["cot_table"] = bc.slot_table(lay.views(state["cotangent"]))
    if op == "stencil":
        state["out"] = torch.zeros_like(buf)
        state["out_table"] = bc.slot_table(lay.views(state["out"]))
    return state


def run(state):
    op = state["op"]
    if op == "forward":
        state["plan"].apply(state["table"])
        return state["fields"]
    if op == "adjoint":
        state["plan"].adjoint(state["table"])
        return state["fields"]
    if op == "both":
        state["plan"].apply(state["table"])
        state["plan"].adjoint(state["cot_table"])
        return [state["fields"], state["cotangent"]]
    if op == "stencil":
        state["plan"].apply_stencil(state["table"], state["out_table"], STENCIL_27, COEFFS_27)
        return [state["fields"], state["out"]]
    state["pack"].run(state["table"], state["buffer"])
    return state["buffer"]


# ---------------------------------------------------------------------------
# the operator in FP64
# ---------------------------------------------------------------------------
# panel frames: outward normal, directions of the first and second angle;
# panels 0..3 go round the equator (+X, +Y, -X, -Y), 4 is +Z, 5 is -Z
FRAMES = np.array([
    [[1, 0, 0], [0, 1, 0], [0, 0, 1]], [[0, 1, 0], [-1, 0, 0], [0, 0, 1]],
    [[-1, 0, 0], [0, -1, 0], [0, 0, 1]], [[0, -1, 0], [1, 0, 0], [0, 0, 1]],
    [[0, 0, 1], [0, 1, 0], [-1, 0, 0]], [[0, 0, -1], [0, 1, 0], [1, 0, 0]]], np.float64)


def _angle(n, i):
    return -math.pi / 4 + (np.asarray(i, np.float64) + 0.5) * (math.pi / (2 * n))


def _basis(panel, a, b):
    """Unit position and its derivatives along the two angles."""
    nrm, ex, ey = FRAMES[panel]
    f = nrm + np.tan(a)[:, None] * ex + np.tan(b)[:, None] * ey
    size = np.linalg.norm(f, axis=1, keepdims=True)
    r = f / size
    tangent = lambda e, ang: ((e - r * (r @ e)[:, None]) / size  # noqa: E731
                              / np.cos(ang)[:, None] ** 2)
    return r, tangent(ex, a), tangent(ey, b)


def _cell_point(n, panel, i, j):
    return _basis(panel, _angle(n, [i]), _angle(n, [j]))[0][0]


def _angles_on(panel, r):
    nrm, ex, ey = FRAMES[panel]
    return np.arctan2(r @ ex, r @ nrm), np.arctan2(r @ ey, r @ nrm)


def _turn(panel, a, b, nb, aq, bq):
    """(n, 2, 2): covariant components on ``nb`` to those on ``panel``."""
    _, ea, eb = _basis(panel, a, b)
    _, qa, qb = _basis(nb, aq, bq)
    own = np.stack([ea, eb], 1)
    g = np.stack([qa, qb], 1)
    dual = np.linalg.solve(g @ g.transpose(0, 2, 1), g)
    return own @ dual.transpose(0, 2, 1)


def _lagrange(tau, p):
    w = np.ones((len(tau), p))
    for k in range(p):
        for m in range(p):
            if m != k:
                w[:, k] *= (tau - m) / (k - m)
    return w


def _average_weights(tau, p):
    """Weights on the averages of cells [k - 1/2, k + 1/2], k < p, of the
    degree p - 1 polynomial with these averages, evaluated at ``tau``."""
    k = np.arange(p)
    e = np.arange(p)
    moments = ((k[:, None] + 0.5) ** (e + 1) - (k[:, None] - 0.5) ** (e + 1)) / (e + 1)
    return np.asarray(tau)[:, None] ** e @ np.linalg.inv(moments)


def _sphere_links(case, lay):
    n, h, p, nq = case["n"], case["h"], case["p"], case["quad"]
    step = math.pi / (2 * n)
    pair = (1, 2) if case["fields"] == "huv" else None
    links = []
    for panel in range(6):
        for axis in (0, 1):
            for side in (0, 1):
                cells = np.zeros((h * n, 3), np.int64)
                depth = np.repeat(np.arange(h), n)
                cells[:, axis] = n + depth if side else -1 - depth
                cells[:, 1 - axis] = np.tile(np.arange(n), h)
                a, b = _angle(n, cells[:, 0]), _angle(n, cells[:, 1])
                r = _basis(panel, a, b)[0]
                nb = int(np.argmax(FRAMES[:, 0] @ r.mean(0)))
                on = [(x + math.pi / 4) / step - 0.5 for x in _angles_on(nb, r)]
                # the axis of the neighbour on which the ghosts are data rows
                flat = [np.abs(x - np.rint(x)).max() for x in on]
                nrm = int(np.argmin(flat))
                row, t = np.rint(on[nrm]).astype(np.int64), on[1 - nrm]
                if nq:
                    parts = _quad_part(case, panel, nb, nrm, cells, row, t)
                else:
                    snap = np.abs(t - np.rint(t)) < 1e-9
                    start = np.clip(np.floor(t).astype(np.int64) - (p // 2 - 1), 0, n - p)
                    w = _lagrange(np.where(snap, np.rint(t), t) - start, p)
                    cols = np.zeros((len(t), p, 3), np.int64)
                    cols[:, :, nrm] = row[:, None]
                    cols[:, :, 1 - nrm] = start[:, None] + np.arange(p)
                    aq, bq = _angles_on(nb, r)
                    turn = _turn(panel, a, b, nb, aq, bq)
                    parts = (cols, w, turn[:, :, :, None] * w[:, None, None, :])
                cols, w, wv = parts
                dst, src = lay.cell_index(panel, cells), lay.cell_index(nb, cols)
                links.append((panel, 0, dst, nb, 0, src, w))
                if pair:
                    for x in (0, 1):
                        for y in (0, 1):
                            links.append((panel, pair[x], dst, nb, pair[y], src, wv[:, x, y]))
    _, bcs = _grid(case)
    return links + [k for d in bcs if d["kind"] == "csr" for k in _csr_links(d, lay)]


def _quad_part(case, panel, nb, nrm, cells, row, t):
    """Columns, scalar weights and vector weights of reconstruction x
    quadrature rows."""
    n, p, nq = case["n"], case["p"], case["quad"]
    step = math.pi / (2 * n)
    pts, gw = np.polynomial.legendre.leggauss(nq)
    lo = np.zeros((len(t), 2), np.int64)
    lo[:, nrm] = np.clip(row - (p // 2 - 1), 0, n - p)
    lo[:, 1 - nrm] = np.clip(np.floor(t + 1e-9).astype(np.int64) - (p // 2 - 1), 0, n - p)
    w = np.zeros((len(t), p * p))
    wv = np.zeros((len(t), 2, 2, p * p))
    for x, wx in zip(pts, gw):
        for y, wy in zip(pts, gw):
            a = _angle(n, cells[:, 0] + x / 2)
            b = _angle(n, cells[:, 1] + y / 2)
            aq, bq = _angles_on(nb, _basis(panel, a, b)[0])
            fa, fb = ((q + math.pi / 4) / step - 0.5 for q in (aq, bq))
            point = (_average_weights(fb - lo[:, 1], p)[:, :, None]
                     * _average_weights(fa - lo[:, 0], p)[:, None, :]).reshape(len(t), -1)
            point *= wx * wy / 4
            w += point
            wv += _turn(panel, a, b, nb, aq, bq)[..., None] * point[:, None, None, :]
    jj, ii = np.meshgrid(np.arange(p), np.arange(p), indexing="ij")
    cols = np.zeros((len(t), p * p, 3), np.int64)
    cols[:, :, 0] = lo[:, :1] + ii.ravel()
    cols[:, :, 1] = lo[:, 1:] + jj.ravel()
    return cols, w, wv


def _box_cells(lo, hi):
    k, j, i = np.meshgrid(*[np.arange(lo[d], hi[d]) for d in (2, 1, 0)], indexing="ij")
    return np.stack([i.ravel(), j.ravel(), k.ravel()], 1)


def _csr_links(d, lay):
    """One link per entry position and source block of a small CSR box."""
    cells = _box_cells(d["lo"], d["hi"])
    ptr = np.asarray(d["row_ptr"])
    row = np.repeat(np.arange(len(ptr) - 1), np.diff(ptr))
    out = []
    for x, c in enumerate(d["comps"]):
        mine = (row >= x * len(cells)) & (row < (x + 1) * len(cells))
        for sb in np.unique(d["col_block"][mine]):
            for sc in np.unique(d["col_comp"][mine]):
                e = mine & (d["col_block"] == sb) & (d["col_comp"] == sc)
                dst = lay.cell_index(d["block"], cells[row[e] - x * len(cells)])
                src = lay.cell_index(int(sb), np.asarray(d["col_ijk"])[e])
                out.append((d["block"], c, dst, int(sb), int(sc), src[:, None],
                            np.asarray(d["val"])[e][:, None]))
    return out


def _mirror(kind, g, n):
    """Data index that ghost index ``g`` of an n-cell axis copies."""
    if kind == "circular":
        return g % n
    return np.where(g < 0, -1 - g, np.where(g >= n, 2 * n - 1 - g, g))


def _face_links(d, lay):
    b = d["block"]
    blk = lay.blocks[b]
    n, h = blk["n"], blk["h"]
    types = {(f["axis"], f["side"]): f for f in d["faces"]}
    out = []
    for axis in range(3):
        for side in (0, 1):
            f = types.get((axis, side))
            if f is None or f["type"] == "zero" or not h[axis]:
                continue
            lo, hi = [0, 0, 0], list(n)
            lo[axis], hi[axis] = (n[axis], n[axis] + h[axis]) if side else (-h[axis], 0)
            g = _box_cells(lo, hi)
            depth = g[:, axis] - n[axis] if side else -1 - g[:, axis]
            src, sb, w = g.copy(), b, np.ones(len(g))
            if f["type"] == "halo":
                sb, sa = f["src_block"], f["src_axis"]
                along, length = g[:, 1 - axis], n[1 - axis]
                src = np.zeros_like(g)
                src[:, sa] = (lay.blocks[sb]["n"][sa] - 1 - depth) if f["src_side"] else depth
                src[:, 1 - sa] = length - 1 - along if f["flip"] else along
            elif f["type"] == "csr":
                nnz, at = f["nnz"][depth, g[:, 1 - axis]], f["layers"][depth, g[:, 1 - axis]]
                src = np.repeat(g[:, None], at.shape[1], 1)
                src[..., axis] = n[axis] - 1 - at if side else at
                w = f["weights"][depth, g[:, 1 - axis]] * (np.arange(at.shape[1]) < nnz[:, None])
                out.append((b, 0, lay.cell_index(b, g), b, 0, lay.cell_index(b, src), w))
                continue
            else:
                src[:, axis] = _mirror(f["type"], g[:, axis], n[axis])
            out.append((b, 0, lay.cell_index(b, g), sb, 0, lay.cell_index(sb, src)[:, None],
                        w[:, None]))
    return out


def _map_links(d, lay):
    g = _box_cells(d["lo"], d["hi"])
    src = lay.cell_index(d["src_block"], g[:, list(d["perm"])] * d["sign"] + d["offset"])
    dst = lay.cell_index(d["block"], g)
    return [(d["block"], c, dst, d["src_block"], c, src[:, None], np.ones((len(g), 1)))
            for c in d["comps"]]


def _links(case, lay):
    """(links of ghost rows, links of averaged data cells): each link is
    (block, component, cells (n,), source block, source component, cells
    (n, k), weights (n, k))."""
    if case["grid"] == "sphere":
        return _sphere_links(case, lay), []
    _, bcs = _grid(case)
    make = {"faces": _face_links, "map": _map_links, "zero": lambda d, lay: []}
    return ([k for d in bcs if d["kind"] in make for k in make[d["kind"]](d, lay)],
            [k for d in bcs if d["kind"] == "sync" for k in _csr_links(d, lay)])


def _fill(lay, x, links, sync, dev):
    """The forward apply of FP64 values ``x``."""
    y = x.clone()
    for view, blk in zip(lay.views(y), lay.blocks):
        keep = _data(view, blk).clone()
        view.zero_()
        _data(view, blk).copy_(keep)
    for b, c, cells, *_ in sync:
        y[lay.where(b, c, cells, dev)] = 0
    for b, c, cells, sb, sc, cols, w in links + sync:
        acc = 0
        for k in range(cols.shape[1]):
            wk = torch.as_tensor(np.ascontiguousarray(w[:, k]), device=dev)[:, None]
            acc = acc + wk * x[lay.where(sb, sc, cols[:, k], dev)].masked_fill(wk == 0, 0)
        at = lay.where(b, c, cells, dev)
        y.index_put_((at,), acc, accumulate=True)
    return y


def _adjoint(lay, y, links, sync, dev):
    """The adjoint of cotangents ``y``: ghosts and averaged cells give their
    cotangent to the cells they read and become zero."""
    x = y.clone()
    for view, blk in zip(lay.views(x), lay.blocks):
        keep = _data(view, blk).clone()
        view.zero_()
        _data(view, blk).copy_(keep)
    for b, c, cells, *_ in sync:
        x[lay.where(b, c, cells, dev)] = 0
    for b, c, cells, sb, sc, cols, w in links + sync:
        got = y[lay.where(b, c, cells, dev)]
        for k in range(cols.shape[1]):
            wk = torch.as_tensor(np.ascontiguousarray(w[:, k]), device=dev)[:, None]
            x.index_put_((lay.where(sb, sc, cols[:, k], dev),), wk * got, accumulate=True)
    return x


def exact(case, seed):
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    lay = _layout(case)
    op = case["op"]
    buf = _fields(case, lay, seed, dev, ghosts=op == "adjoint").double()
    if op == "pack":
        out = []
        for b, lo, hi in _strips(case, lay.blocks):
            cells = lay.cell_index(b, _box_cells(lo, hi))
            out.append(buf[lay.where(b, 0, cells, dev)].T.reshape(-1))
        return torch.cat(out)
    links, sync = _links(case, lay)
    if op == "adjoint":
        return _adjoint(lay, buf, links, sync, dev)
    filled = _fill(lay, buf, links, sync, dev)
    if op == "forward":
        return filled
    if op == "both":
        cot = _fields(case, lay, seed + 1_000_003, dev, ghosts=True).double()
        return [filled, _adjoint(lay, cot, links, sync, dev)]
    out = torch.zeros_like(filled)
    for f, o, blk in zip(lay.views(filled), lay.views(out), lay.blocks):
        n, h = blk["n"], blk["h"]
        acc = 0
        for (i, j, k), c in zip(STENCIL_27, COEFFS_27):
            acc = acc + c * f[:, :, h[2] + k:h[2] + k + n[2], h[1] + j:h[1] + j + n[1],
                              h[0] + i:h[0] + i + n[0]]
        _data(o, blk).copy_(acc)
    return [filled, out]


def work(case):
    """Ghost values written once, every distinct data value the rows read
    once, row tables (weight and column of an entry) once; the adjoint reads
    and clears the ghosts and updates the distinct data values."""
    lay = _layout(case)
    size = 4 if case["dtype"] == "f32" else 8
    op = case["op"]
    if op == "pack":
        values = sum(math.prod(h - l for l, h in zip(lo, hi)) * lay.blocks[b]["nlevels"]
                     for b, lo, hi in _strips(case, lay.blocks))
        return {"bytes": 2 * values * size, "flops": 0}
    ghosts = sum(blk["ncomp"] * blk["nlevels"] * (math.prod(_full(blk)) - math.prod(blk["n"]))
                 for blk in lay.blocks)
    links, sync = _links(case, lay)
    reads, entries, flops = {}, 0, 0
    averaged = {}
    for b, c, cells, sb, sc, cols, w in links + sync:
        used = cols[w != 0]
        reads.setdefault((sb, sc), []).append(used)
        if cols.shape[1] > 1:
            entries += used.size
        flops += 2 * used.size * lay.blocks[b]["nlevels"]
    for b, c, cells, *_ in sync:
        averaged.setdefault((b, c), []).append(cells)
    count = lambda d: sum(np.unique(np.concatenate(v)).size * lay.blocks[b]["nlevels"]  # noqa: E731
                          for (b, _), v in d.items())
    distinct, mean = count(reads), count(averaged)
    forward = (ghosts + mean + distinct) * size + entries * (size + 4)
    adjoint = 2 * (ghosts + mean + distinct) * size + entries * (size + 4)
    if op == "stencil":
        data = sum(math.prod(blk["n"]) for blk in lay.blocks)
        return {"bytes": (2 * data + ghosts) * size, "flops": 2 * len(COEFFS_27) * data + flops}
    return {"bytes": {"forward": forward, "adjoint": adjoint, "both": forward + adjoint}[op],
            "flops": flops * (2 if op == "both" else 1)}
