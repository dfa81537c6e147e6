"""What is measured: the calls a program makes of this library, from one field on a small
mesh to a field on five million faces, with the sizes of the repository's own workloads
(meshgen.workload), its benchmark and its controller training.

A case is a dict of plain values: what is called ("do"), on which mesh family and size, with
which options.  prepare() builds the mesh and everything else a program holds before the
call; run() is the call.  The paths of pch_trace_paths are not returned by any case: a path's
geometry is unique but its list of points is not (zero-length steps at vertices); the
recording solve behind them is measured through the Voronoi labels.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_1305_1293_gb300 import meshgen, pch

FEATURES, HIDDEN = 24, 64          # the controller network: 24 -> 64 -> 64 -> 64 -> 1


def listed():
    return [
        # the smallest call: one field on the 5,120-face sphere, default options, the result
        # on the host (interactive picking on a decimated model)
        {"name": "small_field", "do": "solve", "mesh": "sphere", "a": 16, "b": 0, "control": "plain", "k": 0, "hops": 0,
         "block": 0, "sources": 1, "out": "host"},
        # a mid-size field from a point inside a face, on a grid that is neither square nor
        # even, with boundary; host result
        {"name": "face_point_ragged", "do": "solve", "mesh": "terrain", "a": 187, "b": 331, "control": "plain", "k": 0,
         "hops": 0, "block": 0, "sources": 0, "out": "host"},
        # the 512 x 512 height field from its centre at the options the autotuner finds for it
        # (a program that tuned once); default options are those of the other plain cases
        {"name": "terrain_tuned", "do": "solve", "mesh": "terrain", "a": 512, "b": 512, "control": "plain", "k": 1572864,
         "hops": 32, "block": 64, "sources": 1, "out": "device"},
        # one field on the million-face torus (irregular triangles), learned control
        {"name": "torus_learned", "do": "solve", "mesh": "torus", "a": 1250, "b": 400, "control": "learned", "k": 0,
         "hops": 64, "block": 128, "sources": 1, "out": "device"},
        # the largest: one field on the 5,242,880-face sphere, the benchmark's configuration
        {"name": "large_field", "do": "solve", "mesh": "bumpy", "a": 9, "b": 0, "control": "learned", "k": 0, "hops": 64,
         "block": 128, "sources": 1, "out": "device"},
        # distance to the nearest of 64 sources (sampling, clustering) on 100,820 faces
        {"name": "nearest_of_64", "do": "solve", "mesh": "sphere", "a": 71, "b": 0, "control": "plain", "k": 0, "hops": 0,
         "block": 0, "sources": 64, "out": "device"},
        # eight fields of one mesh in one launch sequence (a row block of a distance matrix)
        {"name": "eight_sources", "do": "batch", "mesh": "bumpy", "a": 7, "b": 0, "control": "learned", "k": 0, "hops": 64,
         "block": 64, "sources": 8, "meshes": 1, "out": "device"},
        # a collection of uneven meshes, one field each, in one launch sequence
        {"name": "collection", "do": "batch", "mesh": "mixed", "a": 2000, "b": 200000, "control": "plain", "k": 0,
         "hops": 0, "block": 0, "sources": 1, "meshes": 24, "out": "host"},
        # a mesh loaded, one field computed and the mesh released again: what a one-shot
        # command-line use pays, host arrays to host array
        {"name": "load_and_solve", "do": "oneshot", "mesh": "bumpy", "a": 6, "b": 0, "control": "plain", "k": 0, "hops": 0,
         "block": 0, "sources": 1, "out": "host"},
        # nearest-source labels and distances (the solve that records its events)
        {"name": "voronoi_labels", "do": "voronoi", "mesh": "bumpy", "a": 7, "b": 0, "control": "plain", "k": 0, "hops": 0,
         "block": 0, "sources": 48, "out": "host"},
        # level sets of a field on 1,310,720 faces (the field on the device, segments to the host)
        {"name": "contour_lines", "do": "contours", "mesh": "bumpy", "a": 8, "b": 0, "control": "plain", "k": 0, "hops": 0,
         "block": 0, "sources": 1, "out": "host", "levels": 32},
        # one full-batch training step of the selection controller (its data set's size)
        {"name": "controller_step", "do": "train", "n": 31722},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges: sizes over their logarithm, odd ones among them."""
    do = rng.choice(["solve", "solve", "solve", "solve", "batch", "mixed", "oneshot", "voronoi", "contours", "train"])
    if do == "train":
        return {"do": "train", "n": _log_int(rng, 200, 32000)}
    family = rng.choice(["sphere", "terrain", "torus", "bumpy"])
    c = {"do": do, "mesh": family, "b": 0, "control": rng.choice(["plain", "plain", "learned"]), "k": 0, "hops": 0,
         "block": 0, "sources": 1, "out": rng.choice(["host", "device"])}
    if c["control"] == "learned" or rng.random() < 0.3:
        c["hops"], c["block"] = rng.choice([(64, 128), (64, 64), (32, 64)])
        if c["control"] == "plain":
            c["k"] = rng.choice([98304, 393216, 1572864])
    # the default 24,576 windows an iteration are for meshes of up to a few hundred thousand faces
    most = 1300000 if do == "contours" or (do == "solve" and c["hops"]) else 330000 if do == "solve" else 100000
    faces = math.exp(rng.uniform(math.log(2000), math.log(most)))
    if family == "sphere":
        c["a"] = max(8, int(round(math.sqrt(min(faces, 600000) / 20.0))))
    elif family == "bumpy":
        c["a"] = max(3, int(math.log(faces * 1.2 / 20.0, 4)))
    else:                              # grids with sides up to 3 : 1
        ratio = math.exp(rng.uniform(-0.55, 0.55))
        c["a"] = max(12, int(math.sqrt(faces / 2.0) * ratio))
        c["b"] = max(12, int(math.sqrt(faces / 2.0) / ratio))
    if do == "solve":
        c["sources"] = rng.choice([0, 1, 1, 1, _log_int(rng, 2, 200)])
    elif do == "batch":
        c["sources"], c["meshes"] = rng.randint(2, 12), 1
    elif do == "mixed":
        c.update({"do": "batch", "mesh": "mixed", "a": 2000, "b": _log_int(rng, 10000, 120000), "sources": 1,
                  "meshes": rng.randint(3, 24)})
    elif do == "voronoi":
        c["sources"], c["out"] = _log_int(rng, 2, 200), "host"
    elif do == "contours":
        c["out"], c["levels"] = "host", _log_int(rng, 4, 48)
    elif do == "oneshot":
        c["out"] = "host"
    return c


# ------------------------------------------------------------------------------ inputs
@functools.lru_cache(maxsize=2)
def _unit_sphere(levels):
    m = meshgen.icosphere(levels, 0.0)
    return m.vertices, m.faces


def _bumpy_sphere(levels, seed):
    """Subdivided icosahedron, radius 1 + 5% of a five-octave sum of plane waves."""
    p, faces = _unit_sphere(levels)
    rng = np.random.default_rng([seed, levels])
    u = rng.normal(size=(8, 3))
    u /= np.linalg.norm(u, axis=1, keepdims=True)
    kappa, phi = rng.uniform(2.0, 4.0, 8), rng.uniform(0.0, 2.0 * math.pi, 8)
    x = torch.from_numpy(p).cuda()
    n = torch.zeros(x.shape[0], dtype=torch.float64, device="cuda")
    for o in range(5):
        for j in range(8):
            proj = x[:, 0] * float(u[j, 0]) + x[:, 1] * float(u[j, 1]) + x[:, 2] * float(u[j, 2])
            n += 2.0 ** (-o) * torch.sin((2.0 ** o) * float(kappa[j]) * proj + float(phi[j]))
    v = x * (1.0 + 0.05 * n / n.abs().max())[:, None]
    return v.cpu().numpy(), faces


def _arrays(family, a, b, seed):
    """(vertices, faces) of one seeded mesh of a family."""
    if family == "bumpy":
        return _bumpy_sphere(a, seed)
    if family == "sphere":
        m = meshgen.geodesic_sphere(a, 0.02, seed=seed)
    elif family == "terrain":
        m = meshgen.terrain(a, b, seed=seed)
    else:
        m = meshgen.torus(a, b, seed=seed)
    return m.vertices, m.faces


def _collection(case, seed):
    """Face counts log-uniform in [a, b] (the same for every seed), each a noisy sphere or a
    height field with the seed's own noise."""
    rng = np.random.default_rng([case["meshes"], case["b"]])
    got = []
    for i in range(case["meshes"]):
        f = math.exp(rng.uniform(math.log(case["a"]), math.log(case["b"])))
        if rng.random() < 0.5:
            got.append(_arrays("sphere", max(2, int(round(math.sqrt(f / 20.0)))), 0, seed + 1000 + i))
        else:
            side = max(2, int(round(math.sqrt(f / 2.0))))
            got.append(_arrays("terrain", side, side, seed + 1000 + i))
    return got


def _sources(nv, n, seed):
    return [int(s) for s in np.random.default_rng([seed, 5]).choice(nv, size=n, replace=False)]


def _train_inputs(n, seed):
    """Features, targets and optimiser state of a training run in progress."""
    rng = np.random.default_rng([seed, n])
    sizes = [(HIDDEN, FEATURES), (HIDDEN, HIDDEN), (HIDDEN, HIDDEN), (1, HIDDEN)]
    p = np.concatenate([np.concatenate([rng.normal(0.0, math.sqrt(2.0 / i), o * i), rng.normal(0.0, 0.05, o)])
                        for o, i in sizes]).astype(np.float32)
    x = rng.uniform(0.0, 1.0, (n, FEATURES)).astype(np.float32)
    x[:, 1:17] = np.sort(x[:, 1:17], axis=1)          # cumulative fractions
    x[:, 23] = 1.0
    t = rng.uniform(0.5, 1.0, n).astype(np.float32)
    m = (rng.normal(0.0, 1e-2, p.size)).astype(np.float32)
    v = (rng.uniform(0.5, 2.0, p.size) * 1e-3).astype(np.float32)
    return p, x, t, m, v


def _options(case):
    o = {"control": pch.CONTROL_LEARNED if case["control"] == "learned" else pch.CONTROL_PLAIN, "k": case["k"],
         "hops": case["hops"], "block": case["block"]}
    if case["out"] == "device":
        o["stream"] = torch.cuda.current_stream()
    return o


def prepare(case, seed):
    s = {"case": case}
    if case["do"] == "train":
        p, x, t, m, v = (torch.from_numpy(q).cuda() for q in _train_inputs(case["n"], seed))
        s.update(p=p, x=x, t=t, m=m, v=v, g=torch.empty_like(p), loss=torch.empty(1, device="cuda"))
        return s
    if case["control"] == "learned":
        pch.load_controller()
    s["options"] = _options(case)
    if case["mesh"] == "mixed":
        arrays = _collection(case, seed)
        s["meshes"] = [pch.Mesh(v, f) for v, f in arrays]
        s["sources"] = [_sources(v.shape[0], 1, seed + i)[0] for i, (v, _) in enumerate(arrays)]
        if case["out"] == "device":
            s["outs"] = [torch.empty(v.shape[0], dtype=torch.float64, device="cuda") for v, _ in arrays]
        return s
    v, f = _arrays(case["mesh"], case["a"], case["b"], seed)
    nv = v.shape[0]
    if case["do"] == "oneshot":
        s.update(v=v, f=f, source=_sources(nv, 1, seed)[0])
        return s
    s["mesh"] = pch.Mesh(v, f)
    if case["do"] == "contours":
        s["field"] = torch.from_numpy(_contour_field(v)).cuda()
        s["levels"] = _contour_levels(_contour_field(v), case["levels"])
        s["segments"] = np.zeros(_contour_room(case), dtype=pch.CONTOUR_DTYPE)
        return s
    if case["do"] == "solve" and case["sources"] == 0:
        rng = np.random.default_rng([seed, 9])
        w = rng.uniform(0.1, 1.0, 3)
        s["face"], s["bary"] = int(rng.integers(f.shape[0])), [float(q) for q in w / w.sum()]
    else:
        s["sources"] = _sources(nv, case["sources"], seed)
    if case["mesh"] == "terrain" and case["sources"] == 1:
        s["sources"] = [meshgen.terrain_center(case["a"], case["b"])]
    if case["do"] == "batch":
        s["meshes"] = [s["mesh"]] * case["sources"]
        if case["out"] == "device":
            s["outs"] = [torch.empty(nv, dtype=torch.float64, device="cuda") for _ in range(case["sources"])]
    elif case["out"] == "device":
        s["out"] = torch.empty(nv, dtype=torch.float64, device="cuda")
    return s


def run(s):
    case = s["case"]
    do = case["do"]
    if do == "train":
        pch.mlp_backward(s["p"], s["x"], s["t"], s["g"], s["loss"], stream=torch.cuda.current_stream())
        pch.mlp_adam(s["p"], s["g"], s["m"], s["v"], 400, 3e-4, stream=torch.cuda.current_stream())
        return {"grad": s["g"], "loss": s["loss"], "params": s["p"], "m": s["m"], "v": s["v"]}
    if do == "batch":
        return pch.solve_batch(s["meshes"], s["sources"], outs=s.get("outs"), **s["options"])
    if do == "oneshot":
        mesh = pch.Mesh(s["v"], s["f"])
        d = pch.solve(mesh, s["source"], **s["options"])
        mesh.close()
        return d
    if do == "voronoi":
        labels, d = pch.voronoi(s["mesh"], s["sources"], **s["options"])
        return {"labels": labels, "dist": d}
    if do == "contours":
        # into the segment buffer that the program draws from
        c = s["segments"]
        got = pch.iso_contours(s["mesh"], s["field"], s["levels"], capacity=len(c))
        c[:len(got)] = got
        return {"level": c["level"], "face": c["face"], "half_edge": c["half_edge"], "t": c["t"]}
    if case["sources"] == 0:
        return pch.solve(s["mesh"], face=s["face"], bary=s["bary"], out=s.get("out"), **s["options"])
    if case["sources"] == 1:
        return pch.solve(s["mesh"], s["sources"][0], out=s.get("out"), **s["options"])
    return pch.solve_multi(s["mesh"], s["sources"], out=s.get("out"), **s["options"])


# ------------------------------------------------------------------------------ work
def _faces(case):
    if case["mesh"] == "bumpy":
        return 20 * 4 ** case["a"]
    if case["mesh"] == "sphere":
        return 20 * case["a"] ** 2
    if case["mesh"] == "mixed":          # mean of a log-uniform count
        return (case["b"] - case["a"]) / math.log(case["b"] / case["a"])
    return 2 * case["a"] * case["b"]


def work(case):
    """Bytes: the mesh's positions and indices, angle and distance state, read and written
    once.  Operations: about 0.4 F^(3/2) windows reach a field's end on these surfaces
    (0.2 on height fields), fewer with more sources, of about 50 FP64 operations each."""
    if case["do"] == "train":
        params = FEATURES * HIDDEN + 2 * HIDDEN * HIDDEN + HIDDEN + 3 * HIDDEN + 1
        return {"bytes": 4.0 * (case["n"] * (FEATURES + 1) + 7 * params), "flops": 6.0 * case["n"] * params}
    f = _faces(case)
    if case["do"] == "contours":
        return {"bytes": 12.0 * f + 4.0 * f + 32.0 * case["levels"] * 2.0 * math.sqrt(f), "flops": 2.0 * f * case["levels"]}
    fields = case["sources"] * 1.0 if case["do"] == "batch" else 1.0
    if case["mesh"] == "mixed":
        fields = case["meshes"] * 1.0
    near = math.sqrt(case["sources"]) if case["do"] in ("solve", "voronoi") and case["sources"] > 1 else 1.0
    windows = (0.2 if case["mesh"] == "terrain" else 0.4) * f ** 1.5 / near
    return {"bytes": fields * (12.0 * f + 24.0 * f / 2 + 8.0 * f / 2), "flops": fields * windows * 50.0}


# ------------------------------------------------------------------------------ 64-bit values
def _contour_field(v):
    """A distance field on the mesh: straight distance from vertex 0 (contours of any field)."""
    d = v - v[0]
    return np.sqrt((d * d).sum(1))


def _contour_levels(field, n):
    return (np.arange(1, n + 1) / (n + 1.0)) * float(field.max())


def _contour_room(case):
    """Segments a program makes room for: a level line crosses a few times sqrt(F) faces."""
    return int(case["levels"] * 6.0 * math.sqrt(_faces(case)))


def exact(case, seed):
    """The controller's training step and the contours in plain numpy, 64 bits.  An exact
    geodesic field in plain numpy takes minutes even on the smallest mesh: None."""
    if case["do"] == "train":
        return _exact_step(*(q.astype(np.float64) for q in _train_inputs(case["n"], seed)))
    if case["do"] != "contours":
        return None
    v, f = _arrays(case["mesh"], case["a"], case["b"], seed)
    field = _contour_field(v)
    levels = _contour_levels(field, case["levels"])
    d = field[f]
    face, level, he, t = [], [], [], []
    for l, lev in enumerate(levels):
        inside = d < lev
        at = np.nonzero(inside.any(1) & ~inside.all(1))[0]
        i, dd = inside[at], d[at]
        nxt = np.roll(i, -1, axis=1)
        leave, enter = np.argmax(i & ~nxt, axis=1), np.argmax(~i & nxt, axis=1)
        k = np.stack([leave, enter], 1)
        r = np.arange(len(at))[:, None]
        p, q = dd[r, k], dd[r, (k + 1) % 3]
        face.append(at)
        level.append(np.full(len(at), l))
        he.append(3 * at[:, None] + k)
        t.append((lev - p) / (q - p))
    face, level, he, t = (np.concatenate(q) for q in (face, level, he, t))
    room = _contour_room(case)
    order = np.lexsort((level, face))[:room]
    padded = {}
    for name, values, kind in (("level", level, np.int32), ("face", face, np.int32), ("half_edge", he, np.int32),
                               ("t", t, np.float64)):
        padded[name] = np.zeros((room,) + values.shape[1:], dtype=kind)
        padded[name][:len(order)] = values[order]
    return padded


def _exact_step(p, x, t, m, v):
    at, w, b = 0, [], []
    for o, i in ((HIDDEN, FEATURES), (HIDDEN, HIDDEN), (HIDDEN, HIDDEN), (1, HIDDEN)):
        w.append(p[at:at + o * i].reshape(o, i))
        b.append(p[at + o * i:at + o * i + o])
        at += o * i + o
    h = [x]
    for q in range(3):
        h.append(np.maximum(h[-1] @ w[q].T + b[q], 0.0))
    e = (h[3] @ w[3].T + b[3])[:, 0] - t
    d = (e / len(t))[:, None]
    parts = []
    for q in (3, 2, 1, 0):
        parts.append(np.concatenate([(d.T @ h[q]).ravel(), d.sum(0)]))
        if q:
            d = (d @ w[q]) * (h[q] > 0.0)
    g = np.concatenate(parts[::-1])
    b1, b2 = float(np.float32(0.9)), float(np.float32(0.999))
    m2 = b1 * m + (1.0 - b1) * g
    v2 = b2 * v + (1.0 - b2) * g * g
    lr = float(np.float32(3e-4))
    step = lr * (m2 / (1.0 - b1 ** 400)) / (np.sqrt(v2 / (1.0 - b2 ** 400)) + 1e-8)
    return {"grad": g, "loss": np.array([0.5 * float((e * e).mean())]), "params": p - step, "m": m2, "v": v2}
