"""The calls that users of this framework make, as timed cases.

Each case goes through the Python binding's public entry points (cga.py; the
planes' array views through the C ABI's cga2d_view) on seeded synthetic clouds
of the kinds and sizes that the repository's own benchmark configurations and
tests use:

  uniform  points uniform in the unit cube (the plain configuration)
  lidar    one spinning-sensor sweep, 64 beams, 256 m grid (frames, sets of
           frames, the pool clouds of the served loop)
  surface  superellipsoid surfaces in a 100 m cube (the 30M-point world and
           the frames of the compression pieces)

Results whose length depends on the data (voxels, planes, neighbour lists,
labels) land in buffers of the largest possible length that the program keeps,
filled with -1 beforehand, as a program with a memory budget holds them: a CGA
as its decoded voxels (the lossless inverse of the build, in CGA order).

Every output is whole numbers (coordinates, indices, squared distances,
labels, bytes): they are compared for equality, so `exact` has no value to add.
"""
from __future__ import annotations

import ctypes
import math

import torch

from paper_2110_11616_gb300 import cga, synth, synth_gpu

# Voxels that a scene can occupy (for the minimal bytes of a pass): the
# 200-object surfaces at 12 bits, a sweep's surroundings at 16 bits.
SURFACE_VOXELS_12 = 31.0e6
LIDAR_VOXELS_16 = 1.75e6


def listed():
    return [
        # The plain configuration: a 100k-point cloud and its moved twin, every
        # operation once.  Some 60 launches of a few microseconds each: what
        # counts is launches, allocations and waits.
        {"name": "plain_step", "op": "step", "kind": "uniform", "n": 100_000, "bits": 10,
         "m": 10_000},
        # One LiDAR sweep brought into the world frame, as it arrives from the
        # sensor ten times a second: a build under a rigid transform.
        {"name": "build_sweep", "op": "build", "kind": "lidar", "n": 131_072, "bits": 16,
         "xform": True},
        # One half of the surface world: the large build.
        {"name": "build_surface", "op": "build", "kind": "surface", "n": 15_000_000, "bits": 12,
         "xform": False},
        # The two halves fused into one world: set union, its three orthogonal
        # projections, decode.
        {"name": "fuse_surface", "op": "fuse", "kind": "surface", "n": 30_000_000, "bits": 12},
        # One small request of the served mix on a resident world (one query
        # to a million; half the requests are below a thousand).
        {"name": "nn_request", "op": "nn", "kind": "lidar", "n": 1_310_720, "bits": 16,
         "m": 1_000, "strategy": "fine"},
        # The frame set's registration queries: a million points near the
        # surfaces of the resident 1.3M-voxel world.
        {"name": "nn_lidar", "op": "nn", "kind": "lidar", "n": 1_310_720, "bits": 16,
         "m": 1_000_000, "strategy": "fine"},
        # The surface world's queries, half on the surfaces and half uniform in
        # the box, with the search structure built for this world (a world is
        # rebuilt every step, so its preparation is part of the pass).
        {"name": "nn_surface", "op": "nn", "kind": "surface", "n": 30_000_000, "bits": 12,
         "m": 4_000_000, "strategy": "tree"},
        # Eight neighbours of every query point (normals, plane fits).
        {"name": "knn_lidar", "op": "knn", "kind": "lidar", "n": 1_310_720, "bits": 16,
         "m": 1_000_000, "k": 8},
        # Every voxel within 10 cm of each query point.
        {"name": "radius_lidar", "op": "radius", "kind": "lidar", "n": 1_310_720, "bits": 16,
         "m": 1_000_000, "r2": 655},
        # Coloured clouds: both halves built with averaged RGB rows and merged.
        {"name": "values_surface", "op": "values", "kind": "surface", "n": 30_000_000, "bits": 12,
         "channels": 3, "policy": "average"},
        # Temporal prediction of a frame: cluster both frames, move the
        # predicted one by its clusters' motion, find each moved voxel's
        # counterpart in the reference.
        {"name": "compress_surface", "op": "compress", "kind": "surface", "n": 30_000_000,
         "bits": 12},
        # Many clouds of mixed size and grid in one planned, graph-replayed
        # pipeline (build, twin, merge, xy projection, 4096 NN queries each), the merged
        # clouds decoded.
        {"name": "batched_mixed", "op": "pipeline", "count": 16, "lo": 5_000, "hi": 2_000_000,
         "m": 4096},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["step", "build", "build", "fuse", "nn", "nn", "knn", "radius", "values",
                     "compress", "pipeline"])
    if op == "step":
        return {"op": op, "kind": "uniform", "n": _log_int(rng, 20_000, 1_000_000),
                "bits": rng.randint(9, 12), "m": _log_int(rng, 500, 50_000)}
    if op == "build":
        if rng.random() < 0.5:
            return {"op": op, "kind": "lidar", "n": _log_int(rng, 20_000, 1_310_720),
                    "bits": rng.randint(13, 16), "xform": True}
        return {"op": op, "kind": "surface", "n": _log_int(rng, 200_000, 15_000_000),
                "bits": rng.randint(10, 13), "xform": rng.random() < 0.3}
    if op == "fuse":
        return {"op": op, "kind": "surface", "n": _log_int(rng, 200_000, 30_000_000),
                "bits": rng.randint(10, 12)}
    if op == "nn":
        if rng.random() < 0.6:
            return {"op": op, "kind": "lidar", "n": _log_int(rng, 100_000, 1_310_720),
                    "bits": rng.randint(14, 16), "m": _log_int(rng, 1, 1_000_000),
                    "strategy": "fine"}
        return {"op": op, "kind": "surface", "n": _log_int(rng, 1_000_000, 30_000_000),
                "bits": rng.randint(11, 12), "m": _log_int(rng, 10_000, 2_000_000),
                "strategy": "tree"}
    if op == "knn":
        k = _log_int(rng, 1, 400)  # up to the neighbourhood of the paper's Fig. 3
        return {"op": op, "kind": "lidar", "n": _log_int(rng, 200_000, 1_310_720),
                "bits": rng.randint(14, 16),
                "m": _log_int(rng, 1_000, min(1_000_000, 20_000_000 // k)), "k": k}
    if op == "radius":
        n, bits, r2 = _log_int(rng, 200_000, 1_310_720), rng.randint(15, 16), _log_int(rng, 50, 1_500)
        most = min(1_000_000, int(21_000_000 / _found(r2, bits, n)))
        return {"op": op, "kind": "lidar", "n": n, "bits": bits, "m": _log_int(rng, 1_000, most),
                "r2": r2}
    if op == "values":
        return {"op": op, "kind": "surface", "n": _log_int(rng, 200_000, 20_000_000),
                "bits": rng.randint(10, 12), "channels": rng.choice([1, 3, 4]),
                "policy": rng.choice(["average", "average", "first"])}
    if op == "compress":
        return {"op": op, "kind": "surface", "n": _log_int(rng, 500_000, 20_000_000),
                "bits": rng.randint(10, 12)}
    return {"op": op, "count": rng.randint(4, 16), "lo": 5_000,
            "hi": _log_int(rng, 50_000, 2_000_000), "m": rng.choice([256, 1000, 4096])}


def _found(r2, bits, n):
    """Mean neighbours per query within sqrt(r2) voxels of a LiDAR world (21 at
    10 cm in the 1.3M-point world on 3.9 mm voxels): as the area of the disc
    and the density of the points."""
    return 21.0 * (r2 / 655.0) * 4.0 ** (16 - bits) * n / 1_310_720


# ------------------------------------------------------------------ inputs
def _cloud(kind, n, seed):
    if kind == "uniform":
        gen = torch.Generator(device="cuda").manual_seed(seed)
        return torch.rand((n, 3), generator=gen, device="cuda", dtype=torch.float32)
    if kind == "lidar":
        return synth_gpu.lidar_cloud(n, seed)
    return synth_gpu.sample_scene(synth_gpu.surface_scene(seed), n, seed + 1)


def _grid(kind, bits):
    if kind == "uniform":
        return cga.grid_from_box([0.0] * 3, 1.0, bits)
    if kind == "lidar":
        return cga.grid_from_box([-128.0] * 3, 256.0, bits)
    return cga.grid_from_box([0.0] * 3, 100.0, bits)


def _frame_motion():
    """1 degree about the scene's vertical axis through its centre, then 0.3 m."""
    c, s = math.cos(math.radians(1.0)), math.sin(math.radians(1.0))
    return [c, -s, 0.0, s, c, 0.0, 0.0, 0.0, 1.0,
            50.0 - (50.0 * c - 50.0 * s) + 0.3, 50.0 - (50.0 * s + 50.0 * c) - 0.2, 0.1]


def _shuffled(points, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    return points[torch.randperm(len(points), generator=gen, device="cuda")].contiguous()


def _kept(shape, dtype):
    return torch.full(shape, -1, dtype=dtype, device="cuda")


def _kept_plane(n, bits):
    """Buffers for one projection of at most n points (h <= 2^bits, g <= 4^bits)."""
    h, g = min(n, 1 << bits), min(n, 1 << (2 * bits))
    return {"U_index": _kept((h,), torch.int16), "U_pointer": _kept((h + 1,), torch.int32),
            "V_index": _kept((g,), torch.int16)}


def prepare(case, seed):
    cga.load()
    op = case["op"]
    s = 10_000 + 101 * int(seed)
    st = {"case": case}
    if op == "pipeline":
        # a third of the way between the two ends of the size range for every
        # three clouds, in the log: a fixed ladder, so that the work of a case
        # does not depend on the seed
        k = case["count"]
        step = math.log(case["hi"] / case["lo"]) / max(k - 1, 1)
        pts, grids, xforms, qs = [], [], [], []
        for i in range(k):
            n = int(case["lo"] * math.exp(step * i)) | 1
            kind = "lidar" if i % 2 == 0 else "surface"
            if kind == "lidar":
                p = synth_gpu.lidar_cloud(n, s + i)
            else:
                p = synth_gpu.surface_cloud(n, s + i, n_objects=max(4, min(200, n // 5000)))
            pts.append(p)
            grids.append(_grid(kind, 10 + (5 * i) % 7))
            xforms.append(synth.rigid_xform(seed=s + 500 + i))
            qs.append(synth_gpu.jitter_queries(p, case["m"], 0.2, s + 1000 + i))
        st["pipe"] = cga.Pipeline(pts, grids, xforms, qs)
        st["pipe"].run_graph()  # captures the graph that every later pass replays
        st["views"] = [st["pipe"].view(i, "merged") for i in range(k)]
        st["xyz"] = [_kept((2 * len(p), 3), torch.int32) for p in pts]
        return st
    kind, n = case["kind"], case["n"]
    grid = st["grid"] = _grid(kind, case["bits"])
    pts = _cloud(kind, n, s)
    if op == "step":
        st["points"], st["twin"] = pts, synth.rigid_xform(seed=s + 3)
        st["queries"] = synth_gpu.uniform_queries(case["m"], s + 4, [0.0] * 3, 1.0)
        st["xyz"] = _kept((2 * n, 3), torch.int32)
        st["planes"] = [_kept_plane(2 * n, case["bits"])]
    elif op == "build":
        st["points"] = pts
        st["xyz"] = _kept((n, 3), torch.int32)
        st["xform"] = None
        if case["xform"]:
            c, v = math.cos(0.02), math.sin(0.02)
            st["xform"] = [c, -v, 0.0, v, c, 0.0, 0.0, 0.0, 1.0, 0.8, -0.4, 0.02]
    elif op == "fuse":
        st["a"] = cga.cga_build(pts[0::2].contiguous(), grid)
        st["b"] = cga.cga_build(pts[1::2].contiguous(), grid)
        st["xyz"] = _kept((n, 3), torch.int32)
        st["planes"] = [_kept_plane(n, case["bits"]) for _ in range(3)]
    elif op in ("nn", "knn", "radius"):
        st["world"] = cga.cga_build(pts, grid)
        if case.get("strategy") == "tree":
            near = synth_gpu.jitter_queries(pts, (case["m"] + 1) // 2, 0.01, s + 5)
            far = synth_gpu.uniform_queries(case["m"] // 2, s + 6, [0.0] * 3, 100.0)
            st["queries"] = torch.cat([near, far]).contiguous()
        else:
            cga.cga_nn_prepare(st["world"])
            st["queries"] = synth_gpu.jitter_queries(pts, case["m"], 0.2, s + 5)
        if op == "radius":
            # the program's room for neighbours: three times the mean
            room = int(3 * _found(case["r2"], case["bits"], n) * case["m"]) + 4096
            st["idx"], st["dist2"] = _kept((room,), torch.int32), _kept((room,), torch.int64)
    elif op == "values":
        gen = torch.Generator(device="cuda").manual_seed(s + 7)
        c = case["channels"]
        base = (pts * 2.55).to(torch.int32)
        noise = torch.randint(-12, 13, (n, c), device="cuda", generator=gen, dtype=torch.int32)
        rows = (base[:, torch.arange(c, device="cuda") % 3] + noise).clamp(0, 255).to(torch.uint8)
        st["points"] = [pts[0::2].contiguous(), pts[1::2].contiguous()]
        st["rows"] = [rows[0::2].contiguous(), rows[1::2].contiguous()]
        st["xyz"] = _kept((n, 3), torch.int32)
        st["merged_rows"] = torch.zeros((n, c), dtype=torch.uint8, device="cuda")
    elif op == "compress":
        st["ref"] = cga.cga_build(pts, grid)
        st["pred"] = cga.cga_build(pts, grid, xform=_frame_motion())
        st["u_ref"], st["u_pred"] = st["ref"].info()["u"], st["pred"].info()["u"]
        # the reference serves every predicted frame of its group
        cga.cga_nn_prepare(st["ref"], "tree")
        st["kept"] = {"ref_labels": torch.zeros(n, dtype=torch.uint8, device="cuda"),
                      "pred_labels": torch.zeros(n, dtype=torch.uint8, device="cuda"),
                      "moved": _kept((n, 3), torch.int32), "idx": _kept((n,), torch.int32),
                      "dist2": _kept((n,), torch.int64)}
    return st


# ------------------------------------------------------------------- passes
class _Cga2dArrays(ctypes.Structure):  # cga2d_arrays of include/cga.h
    _fields_ = [("bits", ctypes.c_uint32), ("plane", ctypes.c_int32), ("h", ctypes.c_uint64),
                ("g", ctypes.c_uint64), ("U_index", ctypes.c_void_p),
                ("U_pointer", ctypes.c_void_p), ("V_index", ctypes.c_void_p)]


class _Borrowed:
    """A device array of a handle, which it keeps alive while a tensor views it."""

    def __init__(self, ptr, count, typestr, owner):
        self.owner = owner
        self.__cuda_array_interface__ = {"shape": (count,), "typestr": typestr,
                                         "data": (ptr, False), "version": 3, "strides": None}


def _keep(out, values):
    """The first len(values) entries of a kept buffer become `values`."""
    out[: len(values)].copy_(values)
    return out


def _keep_plane(out, plane):
    """The three arrays of a projection (int16 and int32 holding the unsigned
    values) into kept buffers."""
    v = _Cga2dArrays()
    rc = cga.load().cga2d_view(plane.ptr, ctypes.byref(v))
    if rc != cga.OK:
        raise cga.CgaError(rc, "cga2d_view")
    for name, ptr, count, typestr in (("U_index", v.U_index, v.h, "<i2"),
                                      ("U_pointer", v.U_pointer, v.h + 1, "<i4"),
                                      ("V_index", v.V_index, v.g, "<i2")):
        _keep(out[name], torch.as_tensor(_Borrowed(ptr, count, typestr, plane), device="cuda"))
    return out


def run(st):
    case = st["case"]
    op = case["op"]
    if op == "step":
        a = cga.cga_build(st["points"], st["grid"])
        b = cga.cga_build(st["points"], st["grid"], xform=st["twin"])
        m = cga.cga_merge(a, b)
        plane = cga.cga_project(m, "xy")
        cga.cga_nn_prepare(m)
        idx, d2 = cga.cga_nn_query(m, st["queries"])
        xyz = cga.cga_decode(m, out=st["xyz"])
        return {"plane": _keep_plane(st["planes"][0], plane), "idx": idx, "dist2": d2, "xyz": xyz}
    if op == "build":
        return cga.cga_decode(cga.cga_build(st["points"], st["grid"], xform=st["xform"]),
                              out=st["xyz"])
    if op == "fuse":
        m = cga.cga_merge(st["a"], st["b"])
        planes = [cga.cga_project(m, p) for p in ("xy", "xz", "yz")]
        xyz = cga.cga_decode(m, out=st["xyz"])
        return {"planes": [_keep_plane(o, p) for o, p in zip(st["planes"], planes)], "xyz": xyz}
    if op == "nn":
        if case["strategy"] == "tree":
            cga.cga_nn_prepare(st["world"], "tree")
        return cga.cga_nn_query(st["world"], st["queries"])
    if op == "knn":
        return cga.cga_knn(st["world"], st["queries"], case["k"])
    if op == "radius":
        offsets, idx, d2 = cga.cga_radius(st["world"], st["queries"], case["r2"])
        return {"offsets": offsets, "idx": _keep(st["idx"], idx), "dist2": _keep(st["dist2"], d2)}
    if op == "values":
        a, b = (cga.cga_build_values(p, r, st["grid"], policy=case["policy"])
                for p, r in zip(st["points"], st["rows"]))
        m = cga.cga_merge_values(a, b, policy="average")
        return {"xyz": cga.cga_decode(m, out=st["xyz"]),
                "rows": _keep(st["merged_rows"], cga.cga_values(m))}
    if op == "compress":
        lr, cr, nr, ir = cga.cga_kmeans(st["ref"], 64, u=st["u_ref"])
        lp, cp, np_, ip = cga.cga_kmeans(st["pred"], 64, u=st["u_pred"])
        mv = cga.cga_motion_vectors(cr, nr, cp, np_)
        moved = cga.cga_reconstruct(st["pred"], lp, mv, u=st["u_pred"])
        idx, d2 = cga.cga_nn_query_voxels(st["ref"], moved)
        kept = st["kept"]
        return {"ref": (_keep(kept["ref_labels"], lr), cr, nr, ir),
                "pred": (_keep(kept["pred_labels"], lp), cp, np_, ip), "mv": mv,
                "moved": _keep(kept["moved"], moved), "idx": _keep(kept["idx"], idx),
                "dist2": _keep(kept["dist2"], d2)}
    pipe = st["pipe"]
    pipe.run_graph()
    return {"merged": [cga.cga_decode(v, out=xyz) for v, xyz in zip(st["views"], st["xyz"])],
            "idx": pipe.idx, "dist2": pipe.dist2}


# ------------------------------------------------------------- minimal work
def _voxels(kind, n, bits):
    """Distinct voxels of a cloud: as many cells as the scene can occupy, drawn
    with replacement."""
    cells = {"surface": SURFACE_VOXELS_12 * 4.0 ** (bits - 12), "uniform": 8.0 ** bits,
             "lidar": LIDAR_VOXELS_16 * 4.0 ** (bits - 16)}[kind]
    return cells * -math.expm1(-n / cells)


def _cga_bytes(kind, u, bits):
    """Z_index (2 B per voxel), Y_index and Y_pointer (6 B per column)."""
    columns = min(u * {"surface": 0.4, "uniform": 0.9, "lidar": 0.9}[kind], 4.0 ** bits)
    return 2.0 * u + 6.0 * columns


def work(case):
    op = case["op"]
    if op == "pipeline":
        step = math.log(case["hi"] / case["lo"]) / max(case["count"] - 1, 1)
        sizes = [int(case["lo"] * math.exp(step * i)) | 1 for i in range(case["count"])]
        n, m = float(sum(sizes)), case["m"] * case["count"]
        # points in; cloud, twin, merged and decoded voxels, the xy plane out; queries
        return {"bytes": 12 * n + 5 * _cga_bytes("lidar", n, 16) + 24 * n + 24.0 * m,
                "flops": 40.0 * n + 8.0 * m}
    kind, n, bits = case["kind"], float(case["n"]), case["bits"]
    u = _voxels(kind, n, bits)
    out = _cga_bytes(kind, u, bits)
    if op == "step":
        u2 = _voxels(kind, 2 * n, bits)
        # points (the twin is the same cloud), decoded voxels, the plane, queries
        return {"bytes": 12 * n + 12 * u2 + 2 * u2 + 24.0 * case["m"],
                "flops": 40.0 * n + 8.0 * case["m"]}
    if op == "build":
        return {"bytes": 12 * n + 12 * u, "flops": (24.0 if case["xform"] else 6.0) * n}
    if op == "fuse":
        half = _voxels(kind, n / 2, bits)
        # both inputs; decoded voxels; three planes of about a column each
        return {"bytes": 2 * _cga_bytes(kind, half, bits) + 12 * u + 3 * 2 * 0.4 * u,
                "flops": 2 * half}
    if op == "nn":
        # a request reads no more of the world than it has queries for
        world = out if case["strategy"] == "tree" else min(out, 64.0 * case["m"])
        return {"bytes": world + 24.0 * case["m"], "flops": 8.0 * case["m"]}
    if op == "knn":
        return {"bytes": out + (12.0 + 12.0 * case["k"]) * case["m"],
                "flops": 8.0 * case["k"] * case["m"]}
    if op == "radius":
        found = _found(case["r2"], bits, n)
        return {"bytes": out + (20.0 + 12.0 * found) * case["m"], "flops": 8.0 * found * case["m"]}
    if op == "values":
        c = case["channels"]
        return {"bytes": (12.0 + c) * n + (12.0 + c) * u, "flops": (6.0 + c) * n}
    # compress: both frames read once, labels, moved voxels and correspondences
    return {"bytes": 2 * out + 2 * u + 24.0 * u, "flops": 2 * 8 * 8.0 * u}


def exact(case, seed):
    return None
