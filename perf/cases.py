"""Timed cases of the collision-response library: what programs have it do.

A cloth or shape solver calls the library once per output frame, with new
positions every time: it detects the edge-face crossings, turns them into
stencils, solves for the displacement, spreads it over the mesh, or asks for
all of that at once (`hfcr_resolve`), for one pair of meshes or for a batch
of pairs.  Each case is one such call on synthetic meshes of the sizes that
the repository's workloads and tests have, from two 1,280-face spheres to a
512 x 512 cloth over a 327,680-face body and 1,024 mesh pairs at once.

The meshes keep their topology from call to call; the positions come from
the case's seed.  `exact` computes the same outputs in float64 with plain
torch: brute-force crossings (culled by boxes), a dense or conjugate-gradient
solve of the stencil system, and the harmonic field by conjugate gradients.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_1409_2081_gb300 import api

DEV = "cuda"
D = 1e-4          # signed distance the response asks for (the library's usual value)
RINGS = 4         # diffusion rings of the frame sequence


# --------------------------------------------------------------------------
# the cases
# --------------------------------------------------------------------------

def listed():
    return [
        # a garment's edge list, derived once per mesh or after remeshing
        {"name": "edges_cloth", "call": "edges", "scene": "cloth", "n": 512},
        # two small bodies in float64: an interactive call, all latency
        {"name": "detect_spheres", "call": "detect", "scene": "spheres", "la": 3, "lb": 3,
         "dtype": "f64", "edges": True, "masses": False},
        # cloth over a torus as a script calls it, the edges left to the library
        {"name": "detect_cloth", "call": "detect", "scene": "cloth_torus", "n": 200, "nu": 256, "nv": 128,
         "dtype": "f32", "edges": False, "masses": False},
        # two 262,144-face closed bodies, both directions
        {"name": "detect_tori", "call": "detect", "scene": "tori", "nu": 512, "nv": 256,
         "dtype": "f32", "edges": True, "masses": False},
        # many independent pairs in one call (a scene of objects, a data set)
        {"name": "detect_batch", "call": "detect_batch", "scene": "batch", "pairs": 1024,
         "lmin": 1, "lmax": 5, "dtype": "f32"},
        # stencils and displacement for a solver that applies them itself
        {"name": "respond_cloth", "call": "respond", "scene": "cloth_torus", "n": 200, "nu": 256, "nv": 128,
         "dtype": "f32", "edges": True, "masses": False},
        # the same on small float64 bodies whose vertices have unequal masses
        {"name": "respond_spheres", "call": "respond", "scene": "spheres", "la": 3, "lb": 3,
         "dtype": "f64", "edges": True, "masses": True},
        # a displacement along a contact curve spread over its vicinity
        {"name": "diffuse_cloth", "call": "diffuse", "scene": "cloth", "n": 512, "rings": RINGS},
        # one response of a small cloth per frame, all latency
        {"name": "frame_small", "call": "frame", "scene": "drape", "n": 41, "level": 3,
         "dtype": "f32", "edges": True, "masses": False, "rings": RINGS, "iters": 1},
        # one response per frame of the large cloth over the large body
        {"name": "frame_large", "call": "frame", "scene": "drape", "n": 512, "level": 7,
         "dtype": "f32", "edges": True, "masses": False, "rings": RINGS, "iters": 1},
        # the repair loop between two small float64 bodies
        {"name": "loop_spheres", "call": "frame", "scene": "spheres", "la": 3, "lb": 3,
         "dtype": "f64", "edges": True, "masses": False, "rings": 0, "iters": 4},
        # one repair iteration of 1,024 pairs at once
        {"name": "frame_batch", "call": "frame_batch", "scene": "batch", "pairs": 1024,
         "lmin": 1, "lmax": 5, "dtype": "f32"},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    call = rng.choice(["edges", "detect", "detect", "detect_batch", "respond", "respond", "diffuse",
                       "frame", "frame", "frame_batch"])
    if call == "edges":
        return {"call": call, "scene": "cloth", "n": _log(rng, 12, 512)}
    if call == "diffuse":
        return {"call": call, "scene": "cloth", "n": _log(rng, 33, 512), "rings": rng.randint(2, 6)}
    if call in ("detect_batch", "frame_batch"):
        return {"call": call, "scene": "batch", "pairs": _log(rng, 8, 1000), "lmin": 1,
                "lmax": rng.randint(3, 5), "dtype": "f32"}
    c = {"call": call, "edges": rng.random() < 0.7, "masses": rng.random() < 0.25}
    scene = rng.choice(["spheres", "cloth_torus", "tori", "drape"] if call != "frame"
                       else ["spheres", "drape", "drape"])
    c["scene"] = scene
    if scene == "spheres":
        c.update(la=rng.randint(2, 5), lb=rng.randint(2, 5), dtype=rng.choice(["f32", "f64"]))
    elif scene == "cloth_torus":
        nu = _log(rng, 48, 256)
        c.update(n=_log(rng, 40, 200), nu=nu, nv=nu // 2 + rng.randint(0, 7), dtype="f32")
    elif scene == "tori":
        nu = _log(rng, 40, 500)
        c.update(nu=nu, nv=nu // 2 + rng.randint(0, 5), dtype="f32")
    else:
        n = _log(rng, 40, 500)
        c.update(n=n, level=min(7, max(3, int(round(math.log2(n / 4.0))))), dtype="f32")
    if call == "frame":
        c.update(rings=RINGS if scene == "drape" else 0, iters=1 if scene == "drape" else rng.randint(1, 4))
    return c


# --------------------------------------------------------------------------
# meshes: topology kept per size, positions from the seed
# --------------------------------------------------------------------------

@functools.lru_cache(maxsize=None)
def _icosphere(level):
    t = (1.0 + math.sqrt(5.0)) / 2.0
    V = np.array([[-1, t, 0], [1, t, 0], [-1, -t, 0], [1, -t, 0], [0, -1, t], [0, 1, t], [0, -1, -t],
                  [0, 1, -t], [t, 0, -1], [t, 0, 1], [-t, 0, -1], [-t, 0, 1]], np.float64)
    V /= np.linalg.norm(V, axis=1, keepdims=True)
    T = np.array([[0, 11, 5], [0, 5, 1], [0, 1, 7], [0, 7, 10], [0, 10, 11], [1, 5, 9], [5, 11, 4],
                  [11, 10, 2], [10, 7, 6], [7, 1, 8], [3, 9, 4], [3, 4, 2], [3, 2, 6], [3, 6, 8],
                  [3, 8, 9], [4, 9, 5], [2, 4, 11], [6, 2, 10], [8, 6, 7], [9, 8, 1]], np.int64)
    for _ in range(level):
        nv = len(V)
        e = np.stack([T, np.roll(T, -1, 1)], 2)               # [m, 3, 2]: ab, bc, ca
        key = e.min(2) * nv + e.max(2)
        uk, inv = np.unique(key.ravel(), return_inverse=True)
        M = V[uk // nv] + V[uk % nv]
        M /= np.linalg.norm(M, axis=1, keepdims=True)
        m = inv.reshape(-1, 3) + nv
        T = np.concatenate([np.stack([T[:, 0], m[:, 0], m[:, 2]], 1), np.stack([T[:, 1], m[:, 1], m[:, 0]], 1),
                            np.stack([T[:, 2], m[:, 2], m[:, 1]], 1), m])
        V = np.concatenate([V, M])
    return V, T.astype(np.int32)


@functools.lru_cache(maxsize=None)
def _torus(nu, nv, R, r):
    u, v = np.meshgrid(2 * np.pi * np.arange(nu) / nu, 2 * np.pi * np.arange(nv) / nv, indexing="ij")
    rho = R + r * np.cos(v)
    V = np.stack([(rho * np.cos(u)).ravel(), (rho * np.sin(u)).ravel(), (r * np.sin(v)).ravel()], 1)
    i, j = np.meshgrid(np.arange(nu), np.arange(nv), indexing="ij")
    i1, j1 = (i + 1) % nu, (j + 1) % nv
    a, b, c, d = (i * nv + j).ravel(), (i1 * nv + j).ravel(), (i1 * nv + j1).ravel(), (i * nv + j1).ravel()
    return V, np.concatenate([np.stack([a, b, c], 1), np.stack([a, c, d], 1)]).astype(np.int32)


@functools.lru_cache(maxsize=None)
def _cloth(n, side):
    s = np.linspace(-side / 2, side / 2, n)
    Y, X = np.meshgrid(s, s, indexing="ij")
    V = np.stack([X.ravel(), Y.ravel(), np.zeros(n * n)], 1)
    i, j = np.meshgrid(np.arange(n - 1), np.arange(n - 1), indexing="ij")
    a = (i * n + j).ravel()
    return V, np.concatenate([np.stack([a, a + 1, a + n + 1], 1),
                              np.stack([a, a + n + 1, a + n], 1)]).astype(np.int32)


def _waves(rng, X, lo, hi, modes=8):
    """A seeded smooth field on the points X, at most 1 in magnitude."""
    f = np.zeros(len(X))
    for _ in range(modes):
        k = rng.standard_normal(X.shape[1])
        k *= rng.uniform(lo, hi) / np.linalg.norm(k)
        f += rng.uniform(0.5, 1.0) * np.sin(X @ k + rng.uniform(0, 2 * np.pi))
    return f / np.abs(f).max()


def _rotation(rng):
    q, r = np.linalg.qr(rng.standard_normal((3, 3)))
    q *= np.sign(np.diag(r))
    return q if np.linalg.det(q) > 0 else -q


def _scene(case, seed):
    """(VA, TA, A oriented, VB, TB, B oriented, segment table or None)."""
    rng = np.random.Generator(np.random.PCG64(seed))
    kind = case["scene"]
    if kind == "spheres":      # two jittered closed spheres, 1.5 radii apart
        VA, TA = _icosphere(case["la"])
        VB, TB = _icosphere(case["lb"])
        VA = VA + rng.uniform(-0.01, 0.01, VA.shape)
        VB = VB + rng.uniform(-0.01, 0.01, VB.shape) + np.array([1.5, 0.0, 0.0])
        return VA, TA, True, VB, TB, True, None
    if kind == "cloth_torus":  # a wavy open cloth cutting into a closed torus
        VA, TA = _cloth(case["n"], 2.0)
        VA = VA.copy()
        VA[:, 2] = 0.4 + 0.3 * _waves(rng, VA[:, :2], 8.0, 24.0)
        VB, TB = _torus(case["nu"], case["nv"], 1.0, 0.4)
        return VA, TA, False, VB, TB, True, None
    if kind == "tori":         # two closed tori overlapping at one place by up to a fifth of the tube
        r = 0.35
        VA, TA = _torus(case["nu"], case["nv"], 1.0, r)
        phi, beta, gamma = rng.uniform(0, 2 * np.pi, 3)
        radial, tangent = np.array([math.cos(phi), math.sin(phi), 0.0]), np.array([-math.sin(phi), math.cos(phi), 0.0])
        u = math.cos(beta) * radial + math.sin(beta) * np.array([0.0, 0.0, 1.0])
        w = math.cos(gamma) * tangent + math.sin(gamma) * np.cross(u, tangent)
        Rm = np.stack([w, np.cross(u, w), u], 1)
        VB = VA @ Rm.T + radial + (2 - rng.uniform(0.05, 0.2)) * r * u - w
        return VA, TA, True, VB, TA, True, None
    if kind == "drape":        # an open cloth lying into the top of a closed bumpy body
        VA, TA = _cloth(case["n"], 3.0)
        VA = VA.copy()
        VA[:, 2] = rng.uniform(0.5, 0.8) + 0.02 * _waves(rng, VA[:, :2], 2.0, 6.0)
        VB, TB = _icosphere(case["level"])
        VB = VB * (1.0 + 0.1 * _waves(rng, VB, 1.0, 8.0))[:, None]
        return VA, TA, False, VB, TB, True, None
    if kind == "batch":        # independent pairs of spheres of uneven sizes, B turned and offset
        out = [[], [], [], []]
        segs = np.zeros((case["pairs"] + 1, 4), np.int64)
        levels = np.random.Generator(np.random.PCG64(case["pairs"])).integers(
            case["lmin"], case["lmax"] + 1, (case["pairs"], 2))   # the same meshes for every seed
        for i in range(case["pairs"]):
            (VA, TA), (VB, TB) = _icosphere(int(levels[i, 0])), _icosphere(int(levels[i, 1]))
            u = rng.standard_normal(3)
            VB = VB @ _rotation(rng).T + rng.uniform(0.5, 1.8) * u / np.linalg.norm(u)
            for lst, x in zip(out, (VA, TA + segs[i, 0], VB, TB + segs[i, 2])):
                lst.append(x)
            segs[i + 1] = segs[i] + (len(VA), len(TA), len(VB), len(TB))
        VA, TA, VB, TB = (np.concatenate(x) for x in out)
        return VA, TA.astype(np.int32), True, VB, TB.astype(np.int32), True, segs.astype(np.int32)
    raise ValueError(kind)


def _masses(case, seed, n):
    """Inverse masses of both meshes between 0.5 and 2, or None."""
    if not case.get("masses"):
        return None, None
    rng = np.random.Generator(np.random.PCG64(seed + 77))
    return tuple(rng.uniform(0.5, 2.0, k).astype(np.float32) for k in n)


def _moved_field(case, seed):
    """A displacement along a closed curve on the cloth (float64 [n, 3]), as a response leaves it."""
    rng = np.random.Generator(np.random.PCG64(seed))
    V, T = _cloth(case["n"], 3.0)
    phi = np.arctan2(V[:, 1], V[:, 0])
    rad = 0.7 + 0.1 * np.sin(3 * phi + rng.uniform(0, 2 * np.pi)) + 0.05 * np.sin(7 * phi + rng.uniform(0, 2 * np.pi))
    on = np.abs(np.hypot(V[:, 0], V[:, 1]) - rad) < 1.6 / (case["n"] - 1)
    return T, np.where(on[:, None], 0.004 * rng.uniform(-1, 1, V.shape), 0.0), V


# --------------------------------------------------------------------------
# prepare and run
# --------------------------------------------------------------------------

def _np_dtype(case):
    return np.float64 if case.get("dtype") == "f64" else np.float32


def _dev(x):
    return torch.from_numpy(np.ascontiguousarray(x)).to(DEV)


def _edge_list(ctx, tris, nv):
    e = torch.empty((3 * tris.shape[0], 2), dtype=torch.int32, device=DEV)
    return e[:ctx.hfcr_build_edges(tris, nv, e)].contiguous()


def _pair_cap(case, VA):
    if case["scene"] == "batch":
        return 2048 * case["pairs"]
    return 1 << 14 if case["scene"] == "spheres" else 1 << 16 if len(VA) < 100_000 else 1 << 18


def prepare(case, seed):
    call = case["call"]
    s = {"call": call, "case": case}
    if call == "edges":
        # vertices numbered strip by strip, the strips in any order
        V, T = _cloth(case["n"], 3.0)
        strip = np.random.Generator(np.random.PCG64(seed)).permutation(case["n"]).astype(np.int32)
        s["tris"], s["nv"] = _dev(strip[T // case["n"]] * case["n"] + T % case["n"]), len(V)
        s["ctx"] = api.Context()
        s["ctx"].hfcr_reserve(len(V), len(T), 16)
        s["out"] = torch.empty((3 * len(T), 2), dtype=torch.int32, device=DEV)
        return s
    if call == "diffuse":
        T, u, V = _moved_field(case, seed)
        s["ctx"] = api.Context()
        s["ctx"].hfcr_reserve(len(V), len(T), 16)
        tris = _dev(T)
        P = _dev(V.astype(np.float32).T)
        s["M"] = api.Mesh(P[0], P[1], P[2], tris, False, edges=_edge_list(s["ctx"], tris, len(V)))
        s["new"] = _dev(u.T)
        s["field"] = torch.empty_like(s["new"])
        return s
    VA, TA, oa, VB, TB, ob, segs = _scene(case, seed)
    nA, nB = len(VA), len(VB)
    # all coordinates in one buffer, so that a frame's new positions are one copy
    P = np.concatenate([VA.T.ravel(), VB.T.ravel()]).astype(_np_dtype(case))
    s["new"] = _dev(P)
    s["pos"] = s["new"].clone()
    x = [s["pos"][i * nA:(i + 1) * nA] for i in range(3)]
    y = [s["pos"][3 * nA + i * nB:3 * nA + (i + 1) * nB] for i in range(3)]
    cap = _pair_cap(case, VA)
    kw = {"diffuse_rings": case["rings"]} if case.get("rings") else {}
    ctx = s["ctx"] = api.Context(**kw)
    ctx.hfcr_reserve(max(nA, nB), max(len(TA), len(TB)), cap)
    ta, tb = _dev(TA), _dev(TB)
    ea = eb = None
    if case.get("edges", True):
        ea, eb = _edge_list(ctx, ta, nA), _edge_list(ctx, tb, nB)
    wa, wb = (None if w is None else _dev(w) for w in _masses(case, seed, (nA, nB)))
    s["A"] = api.Mesh(*x, ta, oa, edges=ea, inv_mass=wa)
    s["B"] = api.Mesh(*y, tb, ob, edges=eb, inv_mass=wb)
    if segs is not None:
        s["segs"] = _dev(segs)
    if call in ("detect", "detect_batch", "respond"):
        s["pairs"] = torch.zeros((cap, 4), dtype=torch.int32, device=DEV)
    if call == "respond":
        s["n"] = ctx.hfcr_detect(s["A"], s["B"], s["pairs"])
        s["st"] = torch.zeros((cap, 4), dtype=torch.int32, device=DEV)
        s["dx"] = torch.zeros_like(s["pos"])
        s["dxA"] = [s["dx"][i * nA:(i + 1) * nA] for i in range(3)]
        s["dxB"] = [s["dx"][3 * nA + i * nB:3 * nA + (i + 1) * nB] for i in range(3)]
    return s


def run(s):
    call, ctx = s["call"], s["ctx"]
    if call == "edges":
        n = ctx.hfcr_build_edges(s["tris"], s["nv"], s["out"])
        return s["out"][:n]
    if call == "diffuse":
        s["field"].copy_(s["new"])           # the frame's displacement
        ctx.hfcr_diffuse(s["M"], s["field"], s["case"]["rings"])
        return s["field"]
    if call == "detect":                     # the pairs are the first n records
        n = ctx.hfcr_detect(s["A"], s["B"], s["pairs"])
        return {"n": n, "pairs": s["pairs"]}
    if call == "detect_batch":
        n = ctx.hfcr_detect_batch(s["A"], s["B"], s["segs"], s["pairs"])
        return {"n": n, "pairs": s["pairs"]}
    if call == "respond":
        k = ctx.hfcr_build_stencils(s["A"], s["B"], s["pairs"], s["n"], s["st"])
        ctx.hfcr_respond(s["A"], s["B"], s["st"], k, D, s["dxA"], s["dxB"])
        return {"k": k, "stencils": s["st"], "dx": s["dx"]}
    s["pos"].copy_(s["new"])                 # the frame's positions
    if call == "frame":
        info = ctx.hfcr_resolve(s["A"], s["B"], D, s["case"]["iters"])
    else:
        info = ctx.hfcr_resolve_batch(s["A"], s["B"], s["segs"], D, 1)
    return {"pos": s["pos"], "iters": info.iters, "pairs": info.total_pairs, "stencils": info.total_stencils}


# --------------------------------------------------------------------------
# what a pass cannot do without
# --------------------------------------------------------------------------

def _sizes(case):
    """Vertices, faces, edges of A and of B."""
    ico = lambda L: (10 * 4 ** L + 2, 20 * 4 ** L, 30 * 4 ** L)  # noqa: E731
    cloth = lambda n: (n * n, 2 * (n - 1) ** 2, 2 * n * (n - 1) + (n - 1) ** 2)  # noqa: E731
    torus = lambda u, v: (u * v, 2 * u * v, 3 * u * v)  # noqa: E731
    k = case["scene"]
    if k == "spheres":
        return ico(case["la"]), ico(case["lb"])
    if k == "cloth":
        return cloth(case["n"]), (0, 0, 0)
    if k == "cloth_torus":
        return cloth(case["n"]), torus(case["nu"], case["nv"])
    if k == "tori":
        return torus(case["nu"], case["nv"]), torus(case["nu"], case["nv"])
    if k == "drape":
        return cloth(case["n"]), ico(case["level"])
    levels = range(case["lmin"], case["lmax"] + 1)     # the expected sizes
    mean = tuple(case["pairs"] * sum(ico(L)[i] for L in levels) / len(levels) for i in range(3))
    return mean, mean


def work(case):
    A, B = _sizes(case)
    es = 8 if case.get("dtype") == "f64" else 4
    call = case["call"]
    if call == "edges":      # triangles in, edges out
        return {"bytes": 12 * A[1] + 8 * A[2], "flops": 0.0}
    if call == "diffuse":    # the field in and out, the edge list in; a ring's mean per band vertex
        return {"bytes": 48 * A[0] + 8 * A[2], "flops": 2.0 * 3 * 7 * A[0]}
    both = case["scene"] not in ("cloth_torus", "drape")   # both directions are tested
    if call == "respond":    # positions of the stencils in, displacements of both meshes out
        return {"bytes": 3 * es * (A[0] + B[0]), "flops": 30.0 * (A[0] + B[0])}
    pos = 3 * es * (A[0] + B[0])
    one = call.startswith("frame") and case.get("iters", 1) == 1   # a single detection tests one direction
    n = 8 * A[2] + 12 * B[1] + ((8 * B[2] + 12 * A[1]) if both and not one else 0)
    if call.startswith("frame"):
        its = case.get("iters", 1)   # the positions are read and written once more per iteration's move
        return {"bytes": pos * (2 + its) + n, "flops": 20.0 * its * (A[2] + B[2])}
    return {"bytes": pos + n, "flops": 20.0 * (A[2] + (B[2] if both else 0))}


# --------------------------------------------------------------------------
# the same results in float64 with plain torch
# --------------------------------------------------------------------------

def _edges64(T):
    e = torch.cat([T[:, [0, 1]], T[:, [1, 2]], T[:, [2, 0]]])
    lo, hi = e.min(1).values, e.max(1).values
    n = int(T.max()) + 1
    k = torch.unique(lo * n + hi)
    return torch.stack([k // n, k % n], 1)


def _orient(a, b, c, p):
    return (torch.linalg.cross(b - a, c - a) * (p - a)).sum(-1)


def _crossings(V, E, W, F, group):
    """(edge, face) ids of the edges of V strictly crossing the faces of W; `group`: edges per culled block."""
    mid = V[E].mean(1)
    ext = (mid.max(0).values - mid.min(0).values).clamp_min(1e-30)
    q = ((mid - mid.min(0).values) / ext * 255).long()
    key = torch.zeros(len(E), dtype=torch.long, device=V.device)
    for b in range(8):
        for c in range(3):
            key |= ((q[:, c] >> b) & 1) << (3 * b + c)
    order = torch.argsort(key, stable=True)
    tri = W[F]
    flo, fhi = tri.min(1).values, tri.max(1).values
    got = []
    for i in range(0, len(E), group):
        e = order[i:i + group]
        p, q2 = V[E[e, 0]], V[E[e, 1]]
        lo, hi = torch.minimum(p, q2), torch.maximum(p, q2)
        near = ((flo <= hi.max(0).values) & (fhi >= lo.min(0).values)).all(1).nonzero()[:, 0]
        if not len(near):
            continue
        box = ((lo[:, None] <= fhi[near][None]) & (hi[:, None] >= flo[near][None])).all(2).nonzero()
        if not len(box):
            continue
        j, f = box[:, 0], near[box[:, 1]]
        a, b, c = tri[f, 0], tri[f, 1], tri[f, 2]
        P, Q = p[j], q2[j]
        s0, s1 = _orient(a, b, c, P), _orient(a, b, c, Q)
        t = torch.stack([_orient(P, Q, a, b), _orient(P, Q, b, c), _orient(P, Q, c, a)])
        hit = (s0 * s1 < 0) & ((t >= 0).all(0) | (t <= 0).all(0))
        got.append(torch.stack([torch.where(s0 < 0, E[e[j], 0], E[e[j], 1])[hit], f[hit], e[j][hit]], 1))
    return torch.cat(got) if got else torch.zeros((0, 3), dtype=torch.long, device=V.device)


def _stencils64(X, T, E, off, dirs, group):
    """Sorted unique stencils [k, 4] of global vertex ids (x0, a, b, c); the number of pairs."""
    rows, n = [], 0
    for d in dirs:
        e, f = (0, 1) if d == 0 else (1, 0)
        h = _crossings(X[off[e]:off[e + 1]], E[e], X[off[f]:off[f + 1]], T[f], group)
        n += len(h)
        u = torch.unique(h[:, :2], dim=0)
        rows.append(torch.cat([u[:, :1] + off[e], T[f][u[:, 1]] + off[f]], 1))
    return torch.cat(rows), n


def _displace64(X, S, minv, d):
    """Displacement of the stencils S at the positions X (None: not solved to float64 accuracy)."""
    dx = torch.zeros_like(X)
    if not len(S):
        return dx
    a, b, c = X[S[:, 1]], X[S[:, 2]], X[S[:, 3]]
    nrm = torch.linalg.cross(b - a, c - a)
    nrm = nrm / nrm.norm(dim=1, keepdim=True)
    rhs = (nrm * (X[S[:, 0]] - (a + b + c) / 3)).sum(1) - d
    coef = torch.tensor([1.0, -1 / 3, -1 / 3, -1 / 3], dtype=X.dtype, device=X.device)
    G = coef[None, :, None] * nrm[:, None]                   # gradient rows [k, 4, 3]
    ids, k = S.reshape(-1), len(S)

    def scatter(lam):
        u = torch.zeros_like(X)
        u.index_add_(0, ids, (G * lam[:, None, None]).reshape(-1, 3))
        return u * minv[:, None]

    def apply(lam):
        return (G * scatter(lam)[S]).sum((1, 2))

    if k <= 10_000:
        A = torch.zeros((k, k), dtype=X.dtype, device=X.device)
        o = torch.argsort(ids, stable=True)
        v, row, role = ids[o], o // 4, o % 4
        _, cnt = torch.unique_consecutive(v, return_counts=True)
        start = torch.cumsum(cnt, 0) - cnt
        left = torch.repeat_interleave(torch.arange(len(v), device=v.device), torch.repeat_interleave(cnt, cnt))
        first = torch.repeat_interleave(torch.repeat_interleave(start, cnt), torch.repeat_interleave(cnt, cnt))
        head = torch.cumsum(torch.repeat_interleave(cnt, cnt), 0) - torch.repeat_interleave(cnt, cnt)
        right = first + torch.arange(len(left), device=v.device) - head[left]
        val = (G[row[left], role[left]] * G[row[right], role[right]]).sum(1) * minv[v[left]]
        A.index_put_((row[left], row[right]), val, accumulate=True)
        L, bad = torch.linalg.cholesky_ex(A)
        if int(bad):
            return None
        lam = torch.cholesky_solve(rhs[:, None], L)[:, 0]
        for _ in range(2):
            lam = lam + torch.cholesky_solve((rhs - apply(lam))[:, None], L)[:, 0]
    else:
        diag = (G.square().sum(2) * minv[S]).sum(1)
        lam, r = torch.zeros_like(rhs), rhs.clone()
        z = r / diag
        p, rz, n0 = z.clone(), (r * z).sum(), rhs.norm()
        for it in range(20000):
            q = apply(p)
            al = rz / (p * q).sum()
            lam, r = lam + al * p, r - al * q
            z = r / diag
            new = (r * z).sum()
            p, rz = z + (new / rz) * p, new
            if it % 100 == 99:
                r = rhs - apply(lam)
                if float(r.norm() / n0) < 1e-13:
                    break
                z = r / diag
                p, rz = z.clone(), (r * z).sum()
        else:
            return None
    return dx - scatter(lam)


def _harmonic64(E, u, fixed, rings):
    """The harmonic field of u on the graph E within `rings` of its nonzero rows; fixed: vertices kept as they are."""
    n = len(u)
    src, dst = torch.cat([E[:, 0], E[:, 1]]), torch.cat([E[:, 1], E[:, 0]])
    reach = (u != 0).any(1)
    moved = reach.clone()
    for _ in range(rings):
        nxt = reach.clone()
        nxt[dst[reach[src]]] = True
        reach = nxt
    band = reach & ~moved & ~fixed
    f = torch.nonzero(band)[:, 0]
    if not len(f):
        return u
    at = torch.full((n,), -1, dtype=torch.long, device=u.device)
    at[f] = torch.arange(len(f), device=u.device)
    deg = torch.bincount(dst, minlength=n)[f].to(u.dtype)[:, None]
    inner = (at[src] >= 0) & (at[dst] >= 0)
    edge = (at[src] < 0) & (at[dst] >= 0)
    rhs = torch.zeros((len(f), 3), dtype=u.dtype, device=u.device).index_add_(0, at[dst[edge]], u[src[edge]])
    i, j = at[src[inner]], at[dst[inner]]
    lap = torch.sparse_coo_tensor(torch.stack([torch.cat([j, at[f]]), torch.cat([i, at[f]])]),
                                  torch.cat([-torch.ones(len(i), dtype=u.dtype, device=u.device), deg[:, 0]]),
                                  (len(f), len(f))).coalesce().to_sparse_csr()
    x = torch.zeros_like(rhs)
    for _ in range(3):                       # conjugate gradients, restarted from the true residual
        r = rhs - lap @ x
        z = r / deg
        p, rz = z.clone(), (r * z).sum(0)
        for _ in range(400):
            q = lap @ p
            al = rz / (p * q).sum(0).clamp_min(1e-300)
            x, r = x + al * p, r - al * q
            z = r / deg
            new = (r * z).sum(0)
            p, rz = z + new / rz.clamp_min(1e-300) * p, new
            if float((r.norm(dim=0) / rhs.norm(dim=0).clamp_min(1e-300)).max()) < 1e-15:
                break
    out = u.clone()
    out[f] = x
    return out


def exact(case, seed):
    call = case["call"]
    if call in ("edges", "detect", "detect_batch"):
        return None                          # whole numbers only
    if call == "diffuse":
        T, u, _ = _moved_field(case, seed)
        E = _edges64(_dev(T.astype(np.int64)))
        none = torch.zeros(len(u), dtype=torch.bool, device=DEV)
        return _harmonic64(E, _dev(u), none, case["rings"]).T.contiguous()
    VA, TA, oa, VB, TB, ob, segs = _scene(case, seed)
    nA, nB = len(VA), len(VB)
    off = [0, nA, nA + nB]
    X = _dev(np.concatenate([VA, VB]).astype(_np_dtype(case)).astype(np.float64))
    T = [_dev(TA.astype(np.int64)), _dev(TB.astype(np.int64))]
    E = [_edges64(t) for t in T]
    wa, wb = _masses(case, seed, (nA, nB))
    minv = torch.ones(nA + nB, dtype=torch.float64, device=DEV) if wa is None else _dev(np.concatenate([wa, wb])).double()
    flat = lambda P: torch.cat([P[:nA].T.reshape(-1), P[nA:].T.reshape(-1)])  # noqa: E731
    both = [0] if not oa else [0, 1]
    if call == "respond":
        S, _ = _stencils64(X, T, E, off, both, 1024)
        dx = _displace64(X, S, minv, D)
        return None if dx is None else {"dx": flat(dx)}
    if call == "frame_batch":
        if case["pairs"] > 64:
            return None                      # over 20 s pair by pair
        rows = []
        for i in range(case["pairs"]):       # pairs are independent: direction 0 of each
            a0, ta, b0, tb = (int(v) for v in segs[i])
            a1, _, b1, tb1 = (int(v) for v in segs[i + 1])
            e = E[0][(E[0][:, 0] >= a0) & (E[0][:, 0] < a1)]
            h = _crossings(X[:nA], e, X[nA:], T[1][tb:tb1], 1024)
            u = torch.unique(h[:, :2], dim=0)
            rows.append(torch.cat([u[:, :1], T[1][u[:, 1] + tb] + nA], 1))
        S = torch.cat(rows)
        dx = _displace64(X, S, minv, D)
        return None if dx is None else {"pos": flat(X + dx)}
    quiet, need = 0, len(both)
    for it in range(case["iters"]):          # the directions take turns
        S, n = _stencils64(X, T, E, off, [both[it % len(both)]], 1024)
        quiet = 0 if n else quiet + 1
        if quiet >= need:
            break
        dx = _displace64(X, S, minv, D)
        if dx is None:
            return None
        if case["rings"]:
            fixed = minv == 0
            for i in range(2):
                sl = slice(off[i], off[i + 1])
                dx[sl] = _harmonic64(E[i], dx[sl], fixed[sl], case["rings"])
        X = X + dx
    return {"pos": flat(X)}
