"""The work that programs have this library do, as measurable cases.

Every case goes through the Python binding's public entry points.  Inputs are
seeded synthetic meshes in the shapes of the library's workloads: tissue
(noisy icosphere nuclei and capped tube vessels), cells around nuclei, a city
of extruded buildings, instanced template meshes and small spheres.  They are
generated in bulk on the device, so that preparing a case costs little more
than loading its meshes and building their BVHs.

Programs keep one context and their datasets with BVHs across calls, so the
states share one context and own their datasets.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2609_24513_gb300 import pierce, synth

QMAX = synth.QMAX
DEV = "cuda" if torch.cuda.is_available() else "cpu"
F64 = torch.float64


# ---------------------------------------------------------------------------
# Cases
# ---------------------------------------------------------------------------

def _join(name, data, n_a, n_b, predicate="intersects", leaf_mode="filtered", width=4, leaf=2,
          cand="boxes", out="host", graph=False):
    return dict(name=name, kind="join", data=data, n_a=n_a, n_b=n_b, predicate=predicate,
                leaf_mode=leaf_mode, width=width, leaf=leaf, cand=cand, out=out, graph=graph)


def listed():
    return [
        # an interactive or scripted call on a handful of small meshes: latency
        # and launches are all there is (the smoke test's shape)
        _join("join_tiny", "spheres", 20, 20, leaf=4),
        # the benchmark's step: every nucleus against every vessel of a slide,
        # resident, replayed from a captured graph, pairs left on the device
        _join("join_tissue_graph", "tissue", 10000, 500, out="device", graph=True),
        # a caller with its own candidate filter: host candidates in, host
        # pairs out, on a medium tissue block of odd size
        _join("join_tissue_host", "tissue", 2311, 117, cand="host"),
        # many placements of resident template meshes (assembly and packing
        # checks): 100,000 translated pairs of very uneven size
        _join("join_instanced", "instanced", 1000, 100000, leaf=4, cand="device", out="device"),
        # precision stress: self join of a city with exactly touching walls;
        # too many pairs to test them all, so the sweep filter runs
        _join("join_urban_self", "urban", 55000, 0),
        # which cell holds which nucleus: the containment predicate
        _join("join_cells_contains", "cells", 6007, 9001, predicate="contains", leaf=4),
        # a loop that must not allocate: caller-owned device buffers
        dict(name="join_noalloc", kind="noalloc", data="tissue", n_a=1501, n_b=75, width=4, leaf=2),
        # the dataset-level formulation with the estimated hashmap
        dict(name="dataset_join", kind="dataset", data="tissue", n_a=1200, n_b=60,
             predicate="intersects", materialize="estimated", width=4, leaf=2, grid=16),
        # the selectivity estimate alone, as a planner calls it
        dict(name="estimate", kind="estimate", data="tissue", n_a=3000, n_b=150, grid=16),
        # datasets in host memory joined cell by cell under a device budget
        dict(name="join_tiled", kind="tiled", data="tissue", n_a=600, n_b=30, grid=2),
        # new data: load from host arrays, build the BVHs, join once, free
        dict(name="load_build_join", kind="load", data="tissue", n_a=700, n_b=35, width=4, leaf=2),
        # serving: a burst of window queries on resident datasets
        dict(name="serve_burst", kind="serve", data="tissue", n_a=4000, n_b=200, n_queries=256),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["join", "join", "join", "join", "noalloc", "dataset", "estimate", "tiled",
                       "load", "serve"])
    width, leaf = rng.choice([2, 4, 4, 8]), rng.choice([1, 2, 2, 4, 8])
    if kind == "join":
        data = rng.choice(["spheres", "tissue", "tissue", "instanced", "urban", "cells"])
        cand = rng.choice(["boxes", "boxes", "host", "device"])
        pred = rng.choice(["intersects", "intersects", "overlap", "contains", "within"])
        if data == "spheres":
            n_a, n_b = _log_int(rng, 8, 300), _log_int(rng, 8, 300)
            pred = rng.choice([pred, "any_vertex"])
        elif data == "tissue":
            n_a = _log_int(rng, 300, 6000)
            n_b = int(n_a * rng.uniform(0.03, 0.06))
        elif data == "instanced":
            n_a, n_b = _log_int(rng, 20, 800), _log_int(rng, 500, 100000)
            cand = rng.choice(["host", "device"])
        elif data == "urban":
            n_a, n_b = _log_int(rng, 200, 50000), 0
            cand = "boxes"
        else:
            n_a, n_b = _log_int(rng, 50, 5000), _log_int(rng, 50, 8000)
        return dict(kind=kind, data=data, n_a=n_a, n_b=n_b, predicate=pred,
                    leaf_mode=rng.choice(["filtered", "filtered", "filtered", "exact"]),
                    width=width, leaf=leaf, cand=cand, out=rng.choice(["host", "device"]),
                    graph=rng.random() < 0.3)
    n_a = _log_int(rng, 400, 1200)
    n_b = int(n_a * rng.uniform(0.04, 0.06))
    if kind == "noalloc":
        return dict(kind=kind, data="tissue", n_a=n_a, n_b=n_b, width=width, leaf=leaf)
    if kind == "dataset":
        data = rng.choice(["tissue", "urban", "spheres"])
        if data == "urban":
            n_a, n_b = _log_int(rng, 200, 20000), 0
        elif data == "spheres":
            n_a, n_b = _log_int(rng, 10, 300), _log_int(rng, 10, 300)
        return dict(kind=kind, data=data, n_a=n_a, n_b=n_b,
                    predicate=rng.choice(["intersects", "overlap"]),
                    materialize=rng.choice(["estimated", "two_pass", "fixed"]),
                    width=width, leaf=leaf, grid=rng.choice([8, 16, 24]))
    if kind == "estimate":
        data = rng.choice(["tissue", "urban", "cells"])
        n_a = _log_int(rng, 50, 2500 if data == "tissue" else 30000)
        n_b = 0 if data == "urban" else max(1, int(n_a * rng.uniform(0.02, 0.06)))
        return dict(kind=kind, data=data, n_a=n_a, n_b=n_b, grid=_log_int(rng, 4, 64))
    if kind == "tiled":
        data = rng.choice(["tissue", "urban"])
        n_a = _log_int(rng, 300, 600) if data == "tissue" else _log_int(rng, 200, 8000)
        n_b = int(n_a * rng.uniform(0.04, 0.06)) if data == "tissue" else 0
        return dict(kind=kind, data=data, n_a=n_a, n_b=n_b, grid=rng.choice([1, 2, 3, 4]))
    if kind == "load":
        data = rng.choice(["tissue", "urban", "cells"])
        if data == "tissue":
            n_a = _log_int(rng, 200, 700)
            n_b = int(n_a * rng.uniform(0.03, 0.06))
        else:
            n_a, n_b = _log_int(rng, 100, 4000), 0 if data == "urban" else _log_int(rng, 100, 4000)
        return dict(kind=kind, data=data, n_a=n_a, n_b=n_b, width=width, leaf=leaf)
    n_a = _log_int(rng, 400, 4000)
    return dict(kind=kind, data="tissue", n_a=n_a, n_b=int(n_a * rng.uniform(0.03, 0.06)),
                n_queries=_log_int(rng, 1, 256))


# ---------------------------------------------------------------------------
# Inputs: meshes in bulk
# ---------------------------------------------------------------------------

class Meshes:
    """Flat arrays of many closed meshes: xyz and tris on the device, offsets
    on the host, per-mesh boxes on the device."""

    def __init__(self, parts):
        xyz, tris, box, nv, nt = [], [], [], [], []
        for V, F in parts:           # V: n x k x 3 grid coordinates, F: f x 3 local ids
            n = V.shape[0]
            if n == 0:
                continue
            V = V.to(torch.float32)
            F = torch.as_tensor(np.ascontiguousarray(F), dtype=torch.int32, device=DEV)
            xyz.append(V.reshape(-1, 3))
            tris.append(F.repeat(n, 1))
            box.append(torch.cat([V.amin(1), V.amax(1)], 1))
            nv += [V.shape[1]] * n
            nt += [F.shape[0]] * n
        self.xyz = torch.cat(xyz).contiguous()
        self.tris = torch.cat(tris).contiguous()
        self.box = torch.cat(box)
        self.voff = np.concatenate([[0], np.cumsum(nv)]).astype(np.int64)
        self.toff = np.concatenate([[0], np.cumsum(nt)]).astype(np.int64)

    @property
    def nmesh(self):
        return len(self.voff) - 1

    def host(self):
        return synth.MeshSet(self.xyz.cpu().numpy(), self.tris.cpu().numpy(), self.voff, self.toff)


def _t(a):
    return torch.as_tensor(np.asarray(a), dtype=F64, device=DEV)


def _quantize(X):
    return torch.clamp(torch.round(X * QMAX), 0, QMAX)


def _noisy_spheres(rng, level, centre, radius, noise):
    """Icospheres of one level with a smooth radial field (8 sinusoids)."""
    U, F = synth.icosphere(level)
    n, parts = len(radius), []
    R = synth.random_rotations(rng, n)
    dirs = rng.normal(size=(n, 8, 3))
    dirs /= np.linalg.norm(dirs, axis=2, keepdims=True)
    w = dirs * rng.uniform(1.0, 3.0, size=(n, 8, 1))
    phase, amp = rng.uniform(0, 2 * np.pi, size=(n, 8)), rng.uniform(0.5, 1.0, size=(n, 8))
    amp = amp / amp.sum(1, keepdims=True) * noise
    U = _t(U)
    step = max(1, 4_000_000 // U.shape[0])
    for k in range(0, n, step):
        s = slice(k, k + step)
        f = torch.zeros(len(radius[s]), U.shape[0], dtype=F64, device=DEV)
        wk, pk, ak = _t(w[s]), _t(phase[s]), _t(amp[s])
        for j in range(8 if noise else 0):
            d = wk[:, None, j, :]
            f += ak[:, j, None] * torch.sin(U[None, :, 0] * d[..., 0] + U[None, :, 1] * d[..., 1] +
                                            U[None, :, 2] * d[..., 2] + pk[:, j, None])
        X = U[None] * (1.0 + f)[..., None]
        Rk = _t(R[s])
        Y = torch.stack([(X * Rk[:, None, i, :]).sum(-1) for i in range(3)], -1)
        parts.append(_quantize(Y * _t(radius[s])[:, None, None] + _t(centre[s])[:, None, :]))
    if not parts:
        return torch.zeros(0, U.shape[0], 3, dtype=F64, device=DEV), F
    return torch.cat(parts), F


def _nuclei(seed, n):
    """Nuclei of a slide: levels 4 and 5, 10 % noise, log-normal radius."""
    rng = np.random.default_rng(seed)
    lev = rng.integers(4, 6, size=n)
    parts = []
    for level in (4, 5):
        m = int((lev == level).sum())
        r = np.clip(np.exp(rng.normal(math.log(1 / 200) - 0.045, 0.3, size=m)), 400 / QMAX, 0.02)
        c = 1.1 * r[:, None] + 2 / QMAX
        c = c + rng.uniform(size=(m, 3)) * (1 - 2 * c)
        parts.append(_noisy_spheres(rng, level, c, r, 0.10))
    return Meshes(parts)


def _tube_faces(rings, sides):
    i, k = np.arange(rings - 1)[:, None], np.arange(sides)[None, :]
    a0, a1 = i * sides + k, i * sides + (k + 1) % sides
    b0, b1 = a0 + sides, a1 + sides
    c0, c1, kk, last = rings * sides, rings * sides + 1, np.arange(sides), (rings - 1) * sides
    return np.concatenate([
        np.stack([a0, a1, b1], -1).reshape(-1, 3), np.stack([a0, b1, b0], -1).reshape(-1, 3),
        np.stack([np.full(sides, c0), (kk + 1) % sides, kk], -1),
        np.stack([np.full(sides, c1), last + kk, last + (kk + 1) % sides], -1)]).astype(np.int32)


def _tubes(rng, n, rings, radius, length, sides=16):
    """Capped tubes around gently winding curves, centred on the origin."""
    d = rng.normal(size=(n, 3))
    d /= np.linalg.norm(d, axis=1, keepdims=True)
    u = np.cross(d, rng.normal(size=(n, 3)))
    u /= np.linalg.norm(u, axis=1, keepdims=True)
    a = rng.uniform(-0.1, 0.1, size=(n, 3, 3)) / np.array([1.0, 4.0, 9.0])[None, :, None]
    t = torch.linspace(0, 1, rings, dtype=F64, device=DEV)[None, :, None]
    d, u, a, length = _t(d), _t(u), _t(a), _t(length)[:, None, None]
    C, T = (t - 0.5) * d[:, None, :], d[:, None, :].expand(n, rings, 3)
    for k in (1, 2, 3):
        C = C + torch.sin(math.pi * k * t) * a[:, k - 1, None, :]
        T = T + math.pi * k * torch.cos(math.pi * k * t) * a[:, k - 1, None, :]
    C, T = C * length, T / T.norm(dim=-1, keepdim=True)
    N = u[:, None, :] - (u[:, None, :] * T).sum(-1, keepdim=True) * T
    N = N / N.norm(dim=-1, keepdim=True)
    B = torch.linalg.cross(T, N)
    th = torch.arange(sides, dtype=F64, device=DEV) * (2 * math.pi / sides)
    ring = C[:, :, None, :] + _t(radius)[:, None, None, None] * (
        torch.cos(th)[:, None] * N[:, :, None, :] + torch.sin(th)[:, None] * B[:, :, None, :])
    V = torch.cat([ring.reshape(n, -1, 3), C[:, :1], C[:, -1:]], 1)
    return V, _tube_faces(rings, sides)


def _vessels(seed, n):
    """Vessels: 16-sided capped tubes of 10,000-50,000 triangles that span
    0.3-1.0 of the slide."""
    rng = np.random.default_rng(seed)
    sizes = [313, 419, 550, 703, 881, 1087, 1312, 1562]
    cls, parts = rng.integers(0, len(sizes), size=n), []
    for k, rings in enumerate(sizes):
        m = int((cls == k).sum())
        r, ext = rng.uniform(1 / 300, 1 / 100, size=m), rng.uniform(0.3, 1.0, size=m)
        at = rng.uniform(size=(m, 3))
        if m == 0:
            continue
        V, F = _tubes(rng, m, rings, r, ext)
        lo, hi = V.amin(1), V.amax(1)
        scale = torch.clamp(0.99 / (hi - lo).amax(1), max=1.0)[:, None, None]
        V, lo, hi = V * scale, lo * scale[:, 0], hi * scale[:, 0]
        room = 0.995 - (hi - lo)
        parts.append((_quantize(V - lo[:, None] + (0.0025 + _t(at) * room)[:, None, :]), F))
    return Meshes(parts)


def _spheres(seed, n, level, r_range, spread):
    rng = np.random.default_rng(seed)
    r = rng.uniform(*r_range, size=n)
    c = 0.5 + spread * rng.uniform(-0.5, 0.5, size=(n, 3))
    return Meshes([_noisy_spheres(rng, level, c, r, 0.0)])


def _cells(seed, n_a, n_b):
    """Cells (A) and nuclei (B), most nuclei well inside a cell, some across
    its wall, the rest elsewhere."""
    rng = np.random.default_rng(seed)
    r = rng.uniform(1 / 120, 1 / 60, size=n_a)
    c = rng.uniform(0.03, 0.97, size=(n_a, 3))
    host = rng.integers(0, n_a, size=n_b)
    s = rng.uniform(0.2, 0.5, size=n_b) * r[host]
    d = rng.normal(size=(n_b, 3))
    d /= np.linalg.norm(d, axis=1, keepdims=True)
    how = rng.choice(3, size=n_b, p=[0.7, 0.2, 0.1])
    off = np.where(how == 0, rng.uniform(0, 0.25, size=n_b), rng.uniform(0.8, 1.1, size=n_b))
    cb = np.where((how == 2)[:, None], rng.uniform(0.03, 0.97, size=(n_b, 3)),
                  c[host] + d * (off * r[host])[:, None])
    half = n_b // 2
    return (Meshes([_noisy_spheres(rng, 4, c, r, 0.08)]),
            Meshes([_noisy_spheres(rng, 3, cb[:half], s[:half], 0.05),
                    _noisy_spheres(rng, 4, cb[half:], s[half:], 0.05)]))


def _prism_faces(n, bands):
    k, kn = np.arange(n), (np.arange(n) + 1) % n
    apex, F = 1 + (bands + 1) * n, []
    F.append(np.stack([np.zeros(n, int), 1 + kn, 1 + k], -1))
    for b in range(bands):
        lo, hi = 1 + b * n, 1 + (b + 1) * n
        F.append(np.stack([lo + k, lo + kn, hi + kn], -1))
        F.append(np.stack([lo + k, hi + kn, hi + k], -1))
    F.append(np.stack([np.full(n, apex), 1 + bands * n + k, 1 + bands * n + kn], -1))
    return np.concatenate(F).astype(np.int32)


def _prisms(foot, z0, height, roof, bands):
    """Closed prisms over integer footprints (m x n x 2), walls in `bands`
    rows, an apex over the footprint's centre."""
    m, n = foot.shape[:2]
    mid = np.rint(foot.mean(1))
    z = np.rint(z0[:, None] + height[:, None] * np.linspace(0, 1, bands + 1))
    V = np.empty((m, 2 + (bands + 1) * n, 3))
    V[:, 0, :2], V[:, 0, 2] = mid, z0
    V[:, 1:-1] = np.concatenate([np.broadcast_to(foot[:, None], (m, bands + 1, n, 2)),
                                 np.broadcast_to(z[:, :, None, None], (m, bands + 1, n, 1))],
                                -1).reshape(m, -1, 3)
    V[:, -1, :2], V[:, -1, 2] = mid, z0 + height + roof
    return np.clip(V, 0, QMAX), _prism_faces(n, bands)


def _urban(seed, n):
    """A city: buildings on a jittered grid (100-2,000 triangles), 5 % of them
    in pairs that touch exactly, and a tenth small boxes and cylinders."""
    rng = np.random.default_rng(seed)
    shapes = [(6, 8), (8, 6), (10, 9), (12, 4), (12, 15), (16, 10), (20, 5), (24, 12), (32, 6),
              (32, 20), (48, 9), (64, 14)]
    n_part = n // 11
    n_pair = int(0.025 * (n - n_part))
    n_star = n - n_part - 2 * n_pair
    side = int(math.ceil(math.sqrt(max(1, n_star + 2 * n_pair))))
    cell = QMAX / (side + 6.0)
    base = rng.permutation(side * side)[:n_star + n_pair]
    base = np.stack([(base % side + 3.5) * cell, (base // side + 3.5) * cell], -1)
    parts = []
    cls = rng.integers(0, len(shapes), size=n_star)
    for k, (sides, bands) in enumerate(shapes):
        at = base[:n_star][cls == k]
        m = len(at)
        th = 2 * np.pi * (np.arange(sides) + rng.uniform(-0.3, 0.3, size=(m, sides))) / sides
        R = cell * rng.uniform(0.35, 0.7, size=m)
        rr = R[:, None] * rng.uniform(0.6, 1.0, size=(m, sides))
        at = at + rng.uniform(-0.2, 0.2, size=(m, 2)) * cell
        foot = np.rint(np.stack([rr * np.cos(th), rr * np.sin(th)], -1) + at[:, None])
        parts.append(_prisms(foot, rng.integers(1000, 3000, size=m).astype(float),
                             np.rint(cell * rng.uniform(0.5, 3, size=m)),
                             np.rint(R * rng.uniform(0.2, 0.5, size=m)), bands))
    # touching pairs: the same rectangle moved by its own width (a shared
    # wall, half a wall, or an edge)
    at, w, h = np.rint(base[n_star:]), int(0.45 * cell), int(0.35 * cell)
    t = np.arange(4) / 4
    rect = np.concatenate([np.stack([w * t, 0 * t], -1), np.stack([w + 0 * t, h * t], -1),
                           np.stack([w - w * t, h + 0 * t], -1), np.stack([0 * t, h - h * t], -1)])
    rect = np.rint(rect)
    z0 = rng.integers(1000, 3000, size=n_pair).astype(float)
    hh = np.rint(cell * rng.uniform(0.5, 3, size=n_pair))
    shift = np.array([[w, 0], [w, h], [w, h // 2]])[rng.integers(0, 3, size=n_pair)]
    for move in (0 * shift, shift):
        parts.append(_prisms(rect[None] + (at + move)[:, None], z0, hh,
                             np.full(n_pair, float(int(0.3 * h))), 3))
    for sides, m in ((4, n_part // 2), (8, n_part // 4), (24, n_part - n_part // 2 - n_part // 4)):
        at = rng.uniform(3 * cell, QMAX - 3 * cell, size=(m, 2))
        th = 2 * np.pi * (np.arange(sides) + 0.5) / sides
        R = rng.uniform(0.1, 0.5, size=m) * cell
        foot = np.rint(R[:, None, None] * np.stack([np.cos(th), np.sin(th)], -1)[None] + at[:, None])
        parts.append(_prisms(foot, np.rint(rng.uniform(800, 3000, size=m)),
                             np.rint(cell * rng.uniform(0.5, 2, size=m)), np.full(m, 4.0), 1))
    return Meshes([(_t(V), F) for V, F in parts])


def _latlong_faces(s, r):
    """Sphere of s segments and r rows: 2 s (r - 1) triangles."""
    j, jn = np.arange(s), (np.arange(s) + 1) % s
    last = 1 + (r - 1) * s
    F = [np.stack([np.zeros(s, int), 1 + j, 1 + jn], -1)]
    for i in range(r - 2):
        a, b = 1 + i * s, 1 + (i + 1) * s
        F.append(np.stack([a + j, b + j, b + jn], -1))
        F.append(np.stack([a + j, b + jn, a + jn], -1))
    F.append(np.stack([np.full(s, last), last - s + jn, last - s + j], -1))
    return np.concatenate(F).astype(np.int32)


def _templates(seed, n):
    """Templates at the cube's centre: noisy spheres and short tubes, 200 to
    50,000 triangles (log-uniform over 12 sizes)."""
    rng = np.random.default_rng(seed)
    sizes = np.exp(np.linspace(math.log(200), math.log(50000), 12))
    cls = rng.integers(0, 12, size=n)
    tube = (rng.random(n) < 0.5) & (sizes[cls] > 1000)
    parts = []
    for k, faces in enumerate(sizes):
        m = int((cls == k)[~tube].sum())
        s = max(3, int(round(math.sqrt(faces / 2))))
        r = max(3, int(round(faces / (2 * s))) + 1)
        lat = np.pi * np.arange(1, r)[:, None] / r
        lon = 2 * np.pi * np.arange(s)[None, :] / s
        U = np.stack([np.sin(lat) * np.cos(lon), np.sin(lat) * np.sin(lon),
                      np.cos(lat) + 0 * lon], -1).reshape(-1, 3)
        U = _t(np.concatenate([[[0, 0, 1.0]], U, [[0, 0, -1.0]]]))
        w, ph = _t(rng.normal(size=(m, 3)) * 2), _t(rng.uniform(0, 6, size=m))
        f = 1 + 0.05 * torch.sin(U[None, :, 0] * w[:, None, 0] + U[None, :, 1] * w[:, None, 1] +
                                 U[None, :, 2] * w[:, None, 2] + ph[:, None])
        rad = _t(rng.uniform(0.01, 0.04, size=m))
        parts.append((_quantize(0.5 + U[None] * f[..., None] * rad[:, None, None]),
                      _latlong_faces(s, r)))
        m = int((cls == k)[tube].sum())
        r, length = rng.uniform(0.003, 0.008, size=m), rng.uniform(0.04, 0.1, size=m)
        if m:
            V, F = _tubes(rng, m, max(2, int(round(faces / 32))), r, length)
            parts.append((_quantize(0.5 + V), F))
    return Meshes(parts)


def _instances(seed, A, B, n):
    """n candidate pairs of templates with translations of B: 30 % across A's
    surface, 10 % deep inside A, the rest with boxes that just overlap."""
    rng = np.random.default_rng(seed)
    ba, bb = A.box.cpu().numpy().astype(np.float64), B.box.cpu().numpy().astype(np.float64)
    ia, ib = rng.integers(0, A.nmesh, size=n), rng.integers(0, B.nmesh, size=n)
    ha, hb = (ba[ia, 3:] - ba[ia, :3]) / 2, (bb[ib, 3:] - bb[ib, :3]) / 2
    d = rng.normal(size=(n, 3))
    d /= np.linalg.norm(d, axis=1, keepdims=True)
    cls = rng.choice(3, size=n, p=[0.3, 0.1, 0.6])[:, None]
    move = np.where(cls == 0, d * ha * rng.uniform(0.85, 1.05, size=(n, 1)),
                    np.where(cls == 1, d * ha * 0.1,
                             rng.choice([-1.0, 1.0], size=(n, 3)) * (ha + hb) *
                             rng.uniform(0.8, 0.95, size=(n, 3))))
    off = np.rint((ba[ia, :3] + ba[ia, 3:]) / 2 + move - (bb[ib, :3] + bb[ib, 3:]) / 2)
    off = np.clip(off, -bb[ib, :3], QMAX - bb[ib, 3:]).astype(np.int32)
    return np.stack([ia, ib], -1).astype(np.int32), off


def _data(case, seed):
    """(A, B or None for a self join) of a case."""
    n_a, n_b = case["n_a"], case["n_b"]
    if case["data"] == "tissue":
        return _nuclei(1000 * seed + 1, n_a), _vessels(1000 * seed + 2, n_b)
    if case["data"] == "spheres":
        spread = 0.5
        return (_spheres(1000 * seed + 3, n_a, 2, (0.05, 0.15), spread),
                _spheres(1000 * seed + 4, n_b, 2, (0.05, 0.15), spread))
    if case["data"] == "cells":
        return _cells(1000 * seed + 5, n_a, n_b)
    if case["data"] == "instanced":
        return _templates(1000 * seed + 6, n_a), _templates(1000 * seed + 7, n_a)
    return _urban(1000 * seed + 8, n_a), None


def _box_pairs(a, b):
    """Pairs of meshes whose closed boxes meet, sorted."""
    got = []
    for k in range(0, a.shape[0], 512):
        x = a[k:k + 512, None]
        ok = ((x[..., :3] <= b[None, :, 3:]) & (b[None, :, :3] <= x[..., 3:])).all(-1)
        p = ok.nonzero()
        p[:, 0] += k
        got.append(p)
    return torch.cat(got).to(torch.int32).contiguous()


# ---------------------------------------------------------------------------
# States
# ---------------------------------------------------------------------------

_ctx = None


def _context():
    global _ctx
    if _ctx is None:
        _ctx = pierce.Context(0)
    return _ctx


class State:
    """A program's handles: its datasets (freed with the state), options and
    the device result it still holds."""

    def __init__(self, case):
        self.case, self.ctx = case, _context()
        self.sets, self.res = [], None

    def add(self, m):
        h = pierce.pj_load_meshes(self.ctx.h, m.xyz, m.tris, m.voff, m.toff)
        self.sets.append(h)
        return h

    def release(self):
        if self.res is not None:
            pierce.pj_free_pairs(self.ctx.h, self.res)
            self.res = None

    def __del__(self):
        try:
            self.release()
            for h in self.sets:
                pierce.pj_free_dataset(self.ctx.h, h)
        except Exception:
            pass


class Pairs:
    """The program's own result buffer: pairs in front, -1 behind them."""

    def __init__(self, n, device=False):
        self.dev = device
        self.buf = torch.full((n, 2), -1, dtype=torch.int32, device=DEV if device else "cpu")
        self.np = None if device else self.buf.numpy()
        self.k = 0

    def put(self, pairs):
        k, to = int(pairs.shape[0]), self.buf if self.dev else self.np
        if k > to.shape[0]:
            raise ValueError("%d pairs, room for %d" % (k, to.shape[0]))
        to[:k] = pairs
        if k < self.k:
            to[k:self.k] = -1
        self.k = k
        return to


class _View:
    def __init__(self, ptr, n):
        self.__cuda_array_interface__ = {"shape": (n, 2), "typestr": "<i4", "data": (ptr, False),
                                         "version": 3}


def prepare(case, seed):
    s = State(case)
    A, B = _data(case, seed)
    s.self_join = B is None
    kind = case["kind"]
    if kind in ("tiled", "load"):        # the program's data is in host memory
        s.A, s.B = A.host(), None if B is None else B.host()
        s.out = Pairs(_room(case))
        return s
    s.out = Pairs(_room(case), case.get("out") == "device")
    s.a = s.add(A)
    s.b = s.a if B is None else s.add(B)
    if kind in ("join", "noalloc", "serve"):
        s.shape = dict(width=case.get("width", 4), leaf_size=case.get("leaf", 2))
        for h in s.sets:
            s.ctx.build(h, s.shape["width"], s.shape["leaf_size"])
    if kind == "join":
        s.cand = s.off = None
        if case["data"] == "instanced":
            s.cand, s.off = _instances(1000 * seed + 9, A, B, case["n_b"])
            if case["cand"] == "device":
                s.cand, s.off = torch.from_numpy(s.cand).to(DEV), torch.from_numpy(s.off).to(DEV)
        elif case["cand"] != "boxes":
            s.cand = _box_pairs(A.box, B.box)
            if case["cand"] == "host":
                s.cand = s.cand.cpu().numpy()
        s.opts = dict(s.shape, predicate=case["predicate"], use_graph=case["graph"],
                      out_host=case["out"] == "host", self_join=s.self_join,
                      leaf_mode=pierce.PJ_LEAF_EXACT if case["leaf_mode"] == "exact"
                      else pierce.PJ_LEAF_FILTERED)
    elif kind == "noalloc":
        s.cand = _box_pairs(A.box, B.box)
        # buffers sized at start-up, for the most candidates it expects
        n = 1024 + int(0.2 * case["n_a"] * case["n_b"])
        if s.cand.shape[0] > n:
            raise ValueError("%d candidates, room for %d" % (s.cand.shape[0], n))
        s.flags = torch.zeros(n, dtype=torch.uint8, device=DEV)
        s.pairs = torch.zeros(n, 2, dtype=torch.int32, device=DEV)
        s.count = torch.zeros(1, dtype=torch.int64, device=DEV)
        s.stream = torch.cuda.current_stream()
    elif kind == "dataset":
        # the dataset BVHs are built by the first call on a dataset and kept
        s.opts = dict(self_join=s.self_join, width=case["width"], leaf_size=case["leaf"],
                      predicate=case["predicate"], materialize=case["materialize"],
                      grid=case["grid"])
        pierce.pj_dataset_join(s.ctx.h, s.a, s.b, **s.opts)
    elif kind == "serve":
        s.lo, s.hi = synth.serving_windows(seed, case["n_queries"])
    return s


def run(s):
    case, ctx = s.case, s.ctx
    kind = case["kind"]
    if kind == "join":
        s.release()
        r = pierce.pj_join_intersects_ex(ctx.h, s.a, s.b, cand=s.cand, cand_offsets=s.off, **s.opts)
        n = int(r.n_candidates)
        if case["out"] == "device":
            s.res = r                     # kept until the next pass
            ptr = pierce.ctypes.cast(r.pairs, pierce.ctypes.c_void_p).value
            got = torch.as_tensor(_View(ptr, int(r.count)), device=DEV) if r.count else s.out.buf[:0]
            return {"pairs": s.out.put(got), "candidates": n}
        pairs = pierce.pairs_to_numpy(r)
        pierce.pj_free_pairs(ctx.h, r)
        return {"pairs": s.out.put(pairs), "candidates": n}
    if kind == "noalloc":
        pierce.pj_join_intersects_noalloc(ctx.h, s.a, s.b, s.cand, s.flags, s.pairs, s.count,
                                          stream=s.stream)
        return {"flags": s.flags, "pairs": s.pairs, "count": s.count}
    if kind == "dataset":
        pairs, _ = pierce.pj_dataset_join(ctx.h, s.a, s.b, **s.opts)
        return s.out.put(pairs)
    if kind == "estimate":
        e = pierce.pj_estimate_join(ctx.h, s.a, s.b, grid=case["grid"], cells=True)
        return {"e_final": e["e_final"], "slots": e["slots"], "cells": e["cells"],
                "occupied": e["cells_occupied"]}
    if kind == "tiled":
        pairs, _ = pierce.pj_join_tiled(ctx.h, s.A, s.B, self_join=s.self_join, grid=case["grid"])
        return s.out.put(pairs)
    if kind == "load":
        a = ctx.load(s.A)
        b = a if s.self_join else ctx.load(s.B)
        for h in {a, b}:
            ctx.build(h, case["width"], case["leaf"])
        pairs, info = ctx.join(a, b, self_join=s.self_join)
        for h in {a, b}:
            pierce.pj_free_dataset(ctx.h, h)
        return {"pairs": s.out.put(pairs), "candidates": info["n_candidates"]}
    tickets = [ctx.submit(s.a, s.b, lo, hi) for lo, hi in zip(s.lo, s.hi)]
    got = [ctx.poll(t)[0] for t in tickets]
    return {"pairs": s.out.put(np.concatenate(got)), "counts": np.array([len(p) for p in got])}


# ---------------------------------------------------------------------------
# Work, tolerances, 64-bit values
# ---------------------------------------------------------------------------

# mean triangles per mesh (A, B) and box-filter candidates
_TRIS = {"tissue": (12800, 27300), "spheres": (320, 320), "cells": (5120, 3200),
         "instanced": (9000, 9000), "urban": (640, 0)}


def _counts(case):
    n_a, n_b = case["n_a"], case["n_b"]
    fa, fb = _TRIS[case["data"]]
    tris = n_a * (fa + fb) if case["data"] == "instanced" else n_a * fa + n_b * fb
    cand = {"tissue": 0.054 * n_a * n_b, "spheres": 0.3 * n_a * n_b, "urban": 1.1 * n_a,
            "cells": 1.2 * n_b + 1e-5 * n_a * n_b, "instanced": n_b}[case["data"]]
    meshes = 2 * n_a if case["data"] == "instanced" else n_a + n_b
    return meshes, tris, max(1.0, cand)


def _room(case):
    """Result pairs a program makes room for (several times what is usual)."""
    n_a, n_b = case["n_a"], case["n_b"]
    n = {"tissue": 256 + 0.002 * n_a * n_b, "spheres": n_a * n_b, "urban": 256 + 3 * n_a,
         "cells": 256 + 3 * n_b + 1e-4 * n_a * n_b, "instanced": n_b}[case["data"]]
    return int(n * (1 + 0.5 * case["n_queries"]) if case["kind"] == "serve" else n)


def work(case):
    meshes, tris, cand = _counts(case)
    mesh_bytes = 18.0 * tris              # 12 B a triangle and 12 B a vertex (half as many)
    kind = case["kind"]
    # a candidate cannot be decided without its pair and both root nodes
    refine = 48.0 * meshes + cand * (8 + 320 + 1)
    if kind in ("join", "noalloc"):
        return {"bytes": refine, "flops": 24.0 * 16 * cand}
    if kind == "dataset":                 # every edge is read and meets at least one node
        return {"bytes": mesh_bytes + tris, "flops": 1.5 * tris * 20}
    if kind == "estimate":
        return {"bytes": mesh_bytes + 24.0 * meshes, "flops": 20.0 * tris}
    if kind in ("tiled", "load"):         # host arrays in, records and nodes out, the join
        return {"bytes": mesh_bytes + tris * (48 + 53) + refine, "flops": 20.0 * tris}
    q = case["n_queries"]                 # a query reads every box; windows hold 14 % on average
    return {"bytes": q * (24.0 * meshes + 0.05 * cand * (8 + 320 + 1)),
            "flops": q * (6.0 * meshes + 0.05 * cand * 24 * 16)}


def tolerance(case):
    # pairs, flags and counts are decided exactly; the estimate is a float64
    # sum whose terms arrive in any order (two runs differ by about 2e-15)
    return {"rel": 1e-13, "max": 1e-12} if case["kind"] == "estimate" else "exact"


def exact(case, seed):
    if case["kind"] != "estimate":
        return None
    A, B = _data(case, seed)
    sides = [A, A if B is None else B]
    G = case["grid"]

    def volume(m):
        toff = torch.as_tensor(m.toff, device=DEV)
        mesh = torch.repeat_interleave(torch.arange(m.nmesh, device=DEV), toff[1:] - toff[:-1])
        voff = torch.as_tensor(m.voff, device=DEV)
        xyz = m.xyz.to(torch.int64)
        tri = m.tris.to(torch.int64) + voff[mesh][:, None]
        a, b, c = (xyz[tri[:, k]] - xyz[voff[mesh]] for k in range(3))
        det = (a * torch.linalg.cross(b, c)).sum(1)      # below 2^59: exact
        return torch.zeros(m.nmesh, dtype=torch.int64, device=DEV).index_add_(0, mesh, det)

    box = [m.box.cpu().numpy().astype(np.float64) / QMAX for m in sides]
    vol = [np.abs(volume(m).cpu().numpy().astype(np.float64)) / 6.0 for m in sides]
    g0 = np.minimum(box[0][:, :3].min(0), box[1][:, :3].min(0))
    g1 = np.maximum(box[0][:, 3:].max(0), box[1][:, 3:].max(0))
    cw = np.maximum(g1 - g0, 1.0 / QMAX) / G
    stat = []
    for b, v in zip(box, vol):
        i0 = np.clip(np.floor((b[:, :3] - g0) / cw), 0, G - 1).astype(int)
        i1 = np.clip(np.floor((b[:, 3:] - g0) / cw), 0, G - 1).astype(int)
        ext = b[:, 3:] - b[:, :3]
        size = ext.prod(1)
        ratio = np.where(size > 0, v / float(QMAX) ** 3 / np.where(size > 0, size, 1), 0.0)
        N, S, R = np.zeros((G, G, G)), np.zeros((G, G, G)), np.zeros((G, G, G))
        for k in range(len(b)):
            at = tuple(slice(i0[k, d], i1[k, d] + 1) for d in range(3))
            N[at] += 1
            S[at] += ext[k].sum() / 3.0
            R[at] += ratio[k]
        stat.append((N, S, R))
    (n1, s1, r1), (n2, s2, r2) = stat
    both = (n1 > 0) & (n2 > 0)
    d1, d2 = np.where(both, n1, 1), np.where(both, n2, 1)
    p = (s1 / d1 + s2 / d2 + 1e-3) ** 3 / cw.prod()
    f = np.sqrt(r1 / d1 * r2 / d2) ** 0.8
    cells = np.where(both, n1 * n2 * np.minimum(p * f, 1.0), 0.0).reshape(-1)
    total = math.fsum(cells)
    return {"e_final": total, "slots": total / 0.5, "cells": cells, "occupied": None}
