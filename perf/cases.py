"""What this framework's users have it do, as measurable cases.

A case is one call (or a short chain of calls) through the package's public entry points on the sizes that the
repository's own workloads, serving stream and tests use: hands of 3, 4 and 5 fingers with 64 or 256 points a link
(or a ragged count), objects of 64^3 to 256^3 voxels or meshes of 2,208 faces, 1 to 256 objects and 1 to 65,536
candidates.  Every pass is ONE optimisation step or evaluation: a longer search in SI units is chaotic at contacts,
so its results could not be compared.  Inputs (hands, objects, candidates) are generated here from the seed alone;
`exact` is plain torch in float64.
"""

from __future__ import annotations

import functools
import math

import numpy as np
import torch

import paper_2306_08132_gb300 as fg

F64 = torch.float64
DEV = "cuda"
M = 7                                           # test velocities: 0, +x, -x, +y, -y, +z, -z


def listed():
    base = {"n_obj": 1, "per_obj": 16, "objects": "superquadric", "grid": 128, "tight": False, "hand": 4, "ppl": 256,
            "r0": 0.010, "mu": 0.5, "w_pen": 0.0, "step": 0, "total": 500}

    def case(name, path, **kw):
        return dict(base, name=name, path=path, **kw)

    return [
        # The smallest call: interactive evaluation of 16 candidates of a 3-finger hand on one small sphere.
        case("grad_tiny", "grad", objects="sphere", grid=64, hand=3, ppl=64, r0=0.004, total=100),
        # One request of the serving stream: a few hundred candidates on one finely sampled object.
        case("grad_one_object", "grad", per_obj=333, objects="polyhedron", grid=256, hand=5),
        # The usual batch: 8 objects, 1,024 initialisations each, one descent step in the middle of the schedule.
        case("step_batch", "step", n_obj=8, per_obj=1024, step=125),
        # The throughput sweep: 256 objects on 192^3 grids (7.2 GB), 65,536 candidates of the 5-finger hand.
        case("step_sweep", "step", n_obj=256, per_obj=256, objects="mixed", grid=192, hand=5, total=1000),
        # The same step from and to pinned host memory, as a planner on the host calls it; an uneven batch.
        case("step_host", "host", n_obj=32, per_obj=509, objects="polyhedron", hand=5, total=100),
        # A user's own torch objective on top: loss and gradient through autograd, a ragged hand (links of 100
        # points), non-cubic grids cropped to the object, the penetration term on.
        case("autograd_ragged", "autograd", n_obj=4, per_obj=777, objects="mixed", grid=97, tight=True, ppl=100,
             w_pen=0.1),
        # The Gauss-Seidel order of the constraint projection, a batch of 8 objects.
        case("gs_batch", "gs", n_obj=8, per_obj=256),
        # The re-queried simulation step (T = 1, as in the paper's experiments).
        case("tstep_batch", "tstep", n_obj=8, per_obj=512, sim_steps=1),
        # Mesh objects (Phong SDF) in the averaged order.
        case("mesh_batch", "grad", n_obj=8, per_obj=128, objects="mesh"),
        # The paper's own combination: mesh objects with the Gauss-Seidel order.
        case("mesh_gs", "gs", n_obj=4, per_obj=128, objects="mesh"),
        # Evaluation of a batch of grasps: contact area and epsilon over 1,024 directions at 5 mm.
        case("quality", "quality", n_obj=8, per_obj=1024, tau=0.005, dirs=1024, edges=8),
        # The stages as single calls for a user's own metric: points, SDF query of all of them, contact wrenches
        # with the contact bits.
        case("stages", "stages", per_obj=2048),
    ]


def draw(rng):
    """A case of the listed ranges (rng: random.Random); sizes spread over their logarithms, odd ones among them."""
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    path = rng.choice(["grad", "step", "step", "host", "autograd", "gs", "tstep", "mesh", "mesh_gs", "quality", "stages"])
    hand = rng.choice([3, 4, 5])
    c = {"path": path, "hand": hand, "ppl": rng.choice([64, 256, 256, rng.randint(48, 256)]), "tight": rng.random() < 0.3,
         "objects": rng.choice(["sphere", "superquadric", "polyhedron", "mixed"]), "grid": rng.choice([64, 128, log_int(33, 256)]),
         "mu": rng.choice([0.5, 0.5, 0.3, 0.8]), "w_pen": rng.choice([0.0, 0.0, 0.1]), "r0": rng.choice([0.004, 0.010]),
         "step": rng.randint(0, 400), "total": 500}
    cap = {"grad": 16384, "step": 16384, "host": 16384, "autograd": 8192, "gs": 2048, "tstep": 4096, "mesh": 1024,
           "mesh_gs": 512, "quality": 8192, "stages": 2048}[path]
    cands = log_int(8, cap)
    c["n_obj"] = 1 if path == "stages" else min(cands, log_int(1, 4 if path == "mesh_gs" else 16))
    c["per_obj"] = max(1, cands // c["n_obj"])
    if path in ("mesh", "mesh_gs"):
        c.update(objects="mesh", path="grad" if path == "mesh" else "gs")
    if path == "tstep":
        c.update(sim_steps=rng.choice([1, 1, 2]), w_pen=0.0)
    if path == "quality":
        c.update(tau=rng.choice([0.005, 0.003, 0.010]), dirs=log_int(64, 2048), edges=rng.choice([4, 8, 8, 12]))
    return c


# --------------------------------------------------------------------------------------------------------- inputs

def _rot(axis, a):
    c, s = math.cos(a), math.sin(a)
    return np.array([[1, 0, 0], [0, c, -s], [0, s, c]]) if axis == "x" else np.array([[c, -s, 0], [s, c, 0], [0, 0, 1]])


def _capsule(length, radius, n):
    """n area-uniform spiral samples of a capsule along +y."""
    a = (np.arange(n) + 0.5) / n
    az = np.arange(n) * math.pi * (3.0 - math.sqrt(5.0))
    fb = radius / (2 * radius + length)                       # one cap's share of the area
    cap, top = a < fb, a >= 1 - fb
    y = np.where(cap, -radius + a / fb * radius, np.where(top, length + (a - 1 + fb) / fb * radius,
                                                          (a - fb) / (1 - 2 * fb) * length))
    h = np.where(cap, y, np.where(top, y - length, 0.0))
    rho = np.sqrt(np.maximum(radius * radius - h * h, 0.0))
    return np.stack([rho * np.cos(az), y, rho * np.sin(az)], -1)


def _box(half, n):
    """n samples of a box's faces, by area."""
    half = np.asarray(half)
    areas = np.repeat([half[1] * half[2], half[0] * half[2], half[0] * half[1]], 2)
    counts = np.floor(areas / areas.sum() * n).astype(int)
    counts[-1] += n - counts.sum()
    out = []
    for f, k in enumerate(counts):
        ax, sign = f // 2, 1 - 2 * (f % 2)
        p = np.empty((k, 3))
        o = [i for i in range(3) if i != ax]
        p[:, ax] = sign * half[ax]
        p[:, o[0]] = (2 * (np.arange(k) + 0.5) / max(k, 1) - 1) * half[o[0]]
        p[:, o[1]] = (2 * ((np.arange(k) * 0.6180339887498949) % 1.0) - 1) * half[o[1]]
        out.append(p)
    return np.concatenate(out)


def _surface_order(p):
    """Points in Morton order, so that neighbours in the list are neighbours on the surface."""
    lo, hi = p.min(0), p.max(0)
    q = ((p - lo) / np.maximum(hi - lo, 1e-12) * 1023).astype(np.int64)
    code = sum(((q[:, a] >> b) & 1) << (3 * b + a) for b in range(10) for a in range(3))
    return np.argsort(code, kind="stable")


@functools.lru_cache(maxsize=32)
def _hand(kind, ppl):
    """Palm box and capsule fingers (3 flexion links each; an abduction knuckle from 4 fingers on; with 5 fingers
    two of them sit on a palm-arch link and the thumb has 5 links): 10, 17 or 23 links."""
    palm = (0.045, 0.045, 0.0125)
    links = [(-1, np.eye(3), np.zeros(3), np.zeros(3), None, (0.0, 0.0))]   # parent, R, o, axis, length, limits

    def finger(root, x, knuckle):
        par, y = root, palm[1]
        if knuckle:
            links.append((par, np.eye(3), np.array([x, y, 0.0]), np.array([0, 0, 1.0]), 0.010, (-0.35, 0.35)))
            par, y = len(links) - 1, y + 0.010
        for ln in (0.045, 0.030, 0.025):
            links.append((par, np.eye(3), np.array([x, y, 0.0]), np.array([1.0, 0, 0]), ln, (0.0, 1.6)))
            par, y = len(links) - 1, y + ln

    xs = (-0.03, 0.0, 0.03) if kind == 3 else (-0.0375, -0.0125, 0.0125, 0.0375)
    for k, x in enumerate(xs):
        if kind == 5 and k == 2:
            links.append((0, np.eye(3), np.array([0.025, 0.005, 0.0]), np.array([0, -1.0, 0]), 0.035, (0.0, 0.5)))
            arch = len(links) - 1
        finger(arch if kind == 5 and k >= 2 else 0, x, kind > 3)
    if kind == 5:
        R = _rot("z", math.radians(50.0)) @ _rot("x", math.radians(20.0))
        par, along = 0, 0.0
        for ax, ln, lim in (((0, 1.0, 0), 0.010, (-0.35, 0.35)), ((0, 0, 1.0), 0.010, (-0.35, 0.35)),
                            ((1.0, 0, 0), 0.035, (0.0, 1.6)), ((1.0, 0, 0), 0.030, (0.0, 1.6)), ((1.0, 0, 0), 0.025, (0.0, 1.6))):
            o = np.array([-palm[0], -0.005, 0.0]) + R @ np.array([0.0, along, 0.0])
            links.append((par, R, o, np.array(ax), ln, lim))
            par, along = len(links) - 1, along + ln
    T, pts, lop, area = [np.eye(3, 4)], [], [], []
    for l, (par, R, o, ax, ln, lim) in enumerate(links):
        if l:
            Rp, op = links[par][1], links[par][2]
            T.append(np.concatenate([Rp.T @ R, (Rp.T @ (o - op))[:, None]], 1))
        s = _box(palm, ppl) if ln is None else _capsule(ln, 0.009, ppl)
        pts.append(s[_surface_order(s)])
        lop += [l] * ppl
        total = 8 * (palm[0] * palm[1] + palm[0] * palm[2] + palm[1] * palm[2]) if ln is None else \
            2 * math.pi * 0.009 * ln + 4 * math.pi * 0.009 ** 2
        area += [total / ppl] * ppl
    f32 = lambda a: np.ascontiguousarray(a, dtype=np.float32)  # noqa: E731
    return {"parent": np.array([x[0] for x in links], np.int32), "T_fix": f32(T), "axis": f32([x[3] for x in links]),
            "q_low": f32([x[5][0] for x in links[1:]]), "q_up": f32([x[5][1] for x in links[1:]]),
            "pts": f32(np.concatenate(pts)), "lop": np.array(lop, np.int32), "area": f32(area),
            "L": len(links), "D": 5 + len(links), "P": ppl * len(links)}


def _nodes(n, pitch, shift):
    ax = [pitch * (torch.arange(n, device=DEV, dtype=torch.float32) - 0.5 * (n - 1) + float(s)) for s in shift]
    return ax[0][None, None, :], ax[1][None, :, None], ax[2][:, None, None]


def _superquadric(rng, n):
    """Radial distance to a superquadric, exponents U(0.3, 2), semi-axes U(2, 8) cm."""
    e1, e2 = rng.uniform(0.3, 2.0, 2)
    a = rng.uniform(0.02, 0.08, 3)
    pitch = (2 * a.max() + 0.04) / (n - 1)
    shift = rng.uniform(-0.5, 0.5, 3)
    x, y, z = _nodes(n, pitch, shift)
    F = ((x / a[0]).abs() ** (2 / e2) + (y / a[1]).abs() ** (2 / e2)) ** (e2 / e1) + (z / a[2]).abs() ** (2 / e1)
    g = (x * x + y * y + z * z).sqrt() * (1.0 - F.clamp(min=1e-30) ** (-e1 / 2))
    return g, pitch, shift, float(a.max()), a


def _sphere(rng, n):
    pitch = 0.126 / (n - 1)
    shift = np.array([0.31, -0.17, 0.23])
    x, y, z = _nodes(n, pitch, shift)
    return (x * x + y * y + z * z).sqrt() - 0.04, pitch, shift, 0.04, np.full(3, 0.04)


def _hull(p):
    """Triangles of the convex hull of a few points in general position: every triple with all others behind it."""
    out = []
    for i in range(len(p)):
        for j in range(i + 1, len(p)):
            for k in range(j + 1, len(p)):
                nrm = np.cross(p[j] - p[i], p[k] - p[i])
                s = (p - p[i]) @ nrm
                if (s <= 1e-12).all():
                    out.append((i, j, k))
                elif (s >= -1e-12).all():
                    out.append((i, k, j))
    return np.array(out)


def _polyhedron(rng, n):
    """Distance to the convex hull of 8 to 22 points on an ellipsoid with semi-axes U(2, 8) cm."""
    k = int(rng.integers(8, 23))
    a = rng.uniform(0.02, 0.08, 3)
    d = rng.normal(size=(k, 3))
    pts = d / np.linalg.norm(d, axis=1, keepdims=True) * a
    shift = rng.uniform(-0.5, 0.5, 3)
    rb = float(np.linalg.norm(pts, axis=1).max())
    pitch = (2 * rb + 0.04) / (n - 1)
    x, y, z = _nodes(n, pitch, shift)
    inside = torch.full((n, n, n), -1e30, device=DEV)
    dist2 = torch.full((n, n, n), 1e30, device=DEV)
    edges = set()
    for tri in _hull(pts):
        v = pts[tri]
        nrm = np.cross(v[1] - v[0], v[2] - v[0])
        nrm /= np.linalg.norm(nrm)
        plane = x * nrm[0] + y * nrm[1] + z * nrm[2] - float(nrm @ v[0])
        inside = torch.maximum(inside, plane)
        in_tri = plane >= 0
        for e in range(3):
            b = np.cross(nrm, v[(e + 1) % 3] - v[e])
            in_tri &= x * b[0] + y * b[1] + z * b[2] >= float(b @ v[e])
            edges.add((min(tri[e], tri[(e + 1) % 3]), max(tri[e], tri[(e + 1) % 3])))
        dist2 = torch.where(in_tri, torch.minimum(dist2, plane * plane), dist2)
    for i, j in sorted(edges):
        e = pts[j] - pts[i]
        t = ((x * e[0] + y * e[1] + z * e[2] - float(e @ pts[i])) / float(e @ e)).clamp(0, 1)
        q = (x - pts[i][0] - t * e[0]) ** 2 + (y - pts[i][1] - t * e[1]) ** 2 + (z - pts[i][2] - t * e[2]) ** 2
        dist2 = torch.minimum(dist2, q)
    g = torch.where(inside < 0, inside, dist2.sqrt())
    return g, pitch, shift, rb, np.abs(pts).max(0)


def _mesh(rng):
    """Superquadric mesh on 24 x 48 latitudes and longitudes (2,208 faces), exponents U(0.5, 1.5)."""
    e1, e2 = rng.uniform(0.5, 1.5, 2)
    a = rng.uniform(0.02, 0.08, 3)
    n_lat, n_lon = 24, 48
    sp = lambda x, e: np.sign(x) * np.abs(x) ** e  # noqa: E731
    eta = -np.pi / 2 + np.pi * np.arange(1, n_lat)[:, None] / n_lat
    om = -np.pi + 2 * np.pi * np.arange(n_lon)[None] / n_lon
    ring = np.stack([a[0] * sp(np.cos(eta), e1) * sp(np.cos(om), e2), a[1] * sp(np.cos(eta), e1) * sp(np.sin(om), e2),
                     a[2] * sp(np.sin(eta), e1) + 0 * om], -1).reshape(-1, 3)
    V = np.concatenate([[[0, 0, -a[2]]], ring, [[0, 0, a[2]]]]).astype(np.float32)
    W, top = V.astype(np.float64), len(V) - 1
    at = lambda i, j: 1 + (i - 1) * n_lon + j % n_lon  # noqa: E731
    F = []
    for j in range(n_lon):
        F += [(0, at(1, j + 1), at(1, j)), (top, at(n_lat - 1, j), at(n_lat - 1, j + 1))]
        for i in range(1, n_lat - 1):
            p, q, s, t = at(i, j), at(i, j + 1), at(i + 1, j), at(i + 1, j + 1)
            nrm = np.cross(W[q] - W[p], W[t] - W[p])                # split a quad so that it folds outwards
            nrm = nrm if nrm @ (W[p] + W[q] + W[t]) > 0 else -nrm
            F += [(p, q, t), (p, t, s)] if nrm @ (W[s] - W[p]) <= 0 else [(p, q, s), (q, t, s)]
    F = np.array(F, np.int32)
    A, B, C = W[F[:, 0]], W[F[:, 1]], W[F[:, 2]]
    flip = (np.cross(B - A, C - A) * (A + B + C)).sum(-1) < 0
    F[flip] = F[flip][:, [0, 2, 1]]
    return {"V": V, "F": F, "rb": float(np.linalg.norm(W, axis=1).max())}


def _objects(case, rng):
    """The case's objects one by one: a generator of dicts.  Beyond 32 shapes the earlier ones come back scaled."""
    kinds = {"mixed": ["superquadric", "polyhedron"]}.get(case["objects"], [case["objects"]])
    shapes = []
    for k in range(case["n_obj"]):
        if kinds[0] == "mesh":
            o = _mesh(rng)
        else:
            if k < 32:
                kind = kinds[k % len(kinds)]
                g, pitch, shift, rb, half = {"sphere": _sphere, "superquadric": _superquadric, "polyhedron": _polyhedron}[kind](rng, case["grid"])
                org = pitch * (shift - 0.5 * (case["grid"] - 1))
                if case["tight"]:                       # the object's box plus 2 cm instead of a cube
                    lo = np.clip(np.floor((-half - 0.02 - org) / pitch).astype(int), 0, case["grid"] - 2)
                    hi = np.clip(np.ceil((half + 0.02 - org) / pitch).astype(int), lo + 1, case["grid"] - 1)
                    g = g[lo[2]:hi[2] + 1, lo[1]:hi[1] + 1, lo[0]:hi[0] + 1].contiguous()
                    org = org + pitch * lo
                shapes.append((g, pitch, org, rb))
                s = 1.0
            else:
                g, pitch, org, rb = shapes[k % 32]
                s = float(rng.uniform(0.8, 1.25))
            o = {"grid": g if s == 1.0 else g * s, "pitch": float(np.float32(pitch * s)), "rb": rb * s,
                 "origin": np.asarray(org * s, dtype=np.float32)}
        o["mass"], o["inertia"] = 1.0, float(np.float32(0.4 * o["rb"] ** 2))
        yield o


def _candidates(case, rng, hand, radii):
    """Palm on a sphere 6 cm outside each object, uniform orientation, joints uniform within their limits."""
    n, per = len(radii) * case["per_obj"], case["per_obj"]
    d = rng.normal(size=(n, 3))
    t = (np.repeat(radii, per) + 0.06)[:, None] * d / np.linalg.norm(d, axis=1, keepdims=True)
    u = rng.normal(size=(n, 4))
    u /= np.linalg.norm(u, axis=1, keepdims=True)
    u *= np.where(u[:, :1] < 0, -1.0, 1.0)
    s = np.linalg.norm(u[:, 1:], axis=1)
    w = u[:, 1:] * (2.0 * np.arctan2(s, u[:, 0]) / np.maximum(s, 1e-12))[:, None]
    th = hand["q_low"] + (hand["q_up"] - hand["q_low"]) * rng.random((n, hand["L"] - 1))
    q = np.concatenate([t, w, th], 1).astype(np.float32)
    return q, np.repeat(np.arange(len(radii)), per).astype(np.int32)


def _params(case):
    return {"alpha_leak": 0.1, "dt": 1e-3, "v_test": 1.0, "mu": case["mu"], "lr": 1e-3, "r0": case["r0"], "w_range": 0.1,
            "w_limit": 1.0, "w_pen": case["w_pen"], "schedule": "linear", "sim_steps": case.get("sim_steps", 0),
            "gauss_seidel": int(case["path"] == "gs")}


def _dilation(case):
    k = np.float32(case["step"]) / np.float32(max(case["total"] - 1, 1))
    return float(max(np.float32(0.0), np.float32(case["r0"]) * (np.float32(1.0) - k)))


def _directions(case, seed):
    u = np.random.default_rng(seed + 77).normal(size=(case["dirs"], 6))
    return (u / np.linalg.norm(u, axis=1, keepdims=True)).astype(np.float32)


def prepare(case, seed):
    rng = np.random.default_rng(seed)
    h = _hand(case["hand"], case["ppl"])
    hand = fg.Hand(h["parent"], h["T_fix"], h["axis"], h["q_low"], h["q_up"], h["pts"], h["lop"])
    sdfs, radii = [], []
    for o in _objects(case, rng):
        sdfs.append(fg.Sdf.from_mesh(o["V"], o["F"], o["mass"], o["inertia"]) if "V" in o else
                    fg.Sdf(o["grid"], o["origin"], o["pitch"], o["mass"], o["inertia"]))
        radii.append(o["rb"])
    q, oc = _candidates(case, rng, h, np.array(radii))
    s = {"case": case, "hand": hand, "scene": fg.Scene(sdfs), "sdf": sdfs[0], "prm": _params(case), "r": _dilation(case),
         "oc": torch.tensor(oc, device=DEV), "q": torch.tensor(q, device=DEV)}
    if case["path"] == "host":
        s["host_in"] = torch.tensor(q).pin_memory()
        s["host_out"] = torch.empty(q.shape).pin_memory()
        s["host_loss"] = torch.empty(len(q)).pin_memory()
    if case["path"] == "quality":
        s["dirs"] = torch.tensor(_directions(case, seed), device=DEV)
        s["area"] = torch.tensor(h["area"], device=DEV)
    return s


def run(s):
    c, hand, scene, q, oc, prm, r = s["case"], s["hand"], s["scene"], s["q"], s["oc"], s["prm"], s["r"]
    if c["path"] == "step":
        x = q.clone()
        loss = fg.optimize_step(hand, scene, x, prm, c["step"], c["total"], 1, obj_of_cand=oc)
        return {"q": x, "loss": loss}
    if c["path"] == "host":
        fg.optimize_step_host(hand, scene, s["host_in"], q, prm, c["step"], c["total"], 1, obj_of_cand=oc,
                              host_q_out=s["host_out"], host_loss=s["host_loss"])
        return {"q": s["host_out"], "loss": s["host_loss"]}
    if c["path"] == "autograd":
        x = q.detach().requires_grad_(True)
        loss = fg.grasp_loss(x, hand, scene, prm, r, obj_of_cand=oc)
        (grad,) = torch.autograd.grad(loss.sum(), x)
        return {"loss": loss, "grad": grad}
    if c["path"] == "quality":
        area = fg.contact_measure(hand, scene, q, s["area"], c["tau"], obj_of_cand=oc)
        eps, n = fg.grasp_epsilon(hand, scene, q, c["tau"], prm["mu"], c["edges"], 12.5, s["dirs"], obj_of_cand=oc)
        return {"area": area, "eps": eps, "contacts": n}
    if c["path"] == "stages":
        pts = fg.fk(hand, q)
        phi, g = fg.sdf_query(s["sdf"], pts, r)
        W, n, bits = fg.contact_wrench(hand, scene, q, prm, r, obj_of_cand=oc, want_bits=True)
        return {"points": pts, "phi": phi, "phi_grad": g, "wrench": W, "contacts": n, "bits": bits}
    loss, grad = fg.loss_and_grad(hand, scene, q, prm, r, obj_of_cand=oc)     # grad, gs, tstep
    return {"loss": loss, "grad": grad}


def work(case):
    """Bytes: the objects, hand and candidates read once, the results written once (an object's grid no more often
    than its cells can be touched: 8 values for each of its points).  Flops: per hand point and pass, the point (18),
    the lookup with its gradient (55), the constraints (12) and, with a gradient, the leaky adjoint of seven
    simulations, of the normal and of the lookup (215: a point out of contact, shared products taken once)."""
    h = _hand(case["hand"], case["ppl"])
    B = case["n_obj"] * case["per_obj"]
    pts = B * h["P"]
    if case["objects"] == "mesh":
        obj = case["n_obj"] * (2208 * 3 * 4 + 1106 * 3 * 4)
    else:
        obj = case["n_obj"] * min(case["grid"] ** 3 * 4, case["per_obj"] * h["P"] * 32)
    byt = obj + h["P"] * 16 + B * (4 * h["D"] + 4)
    if case["path"] == "stages":
        return {"bytes": byt + pts * 28 + B * M * (24 + 4 + 4 * ((h["P"] + 31) // 32)), "flops": pts * (18 + 55 + 12)}
    if case["path"] == "quality":
        return {"bytes": byt + B * 12 + case["dirs"] * 24, "flops": pts * (18 + 40)}
    fl = 300 * pts
    if case["path"] == "tstep":
        fl = pts * (18 + case["sim_steps"] * M * (55 + 60))
    return {"bytes": byt + B * (4 * h["D"] + 4), "flops": fl}


# ------------------------------------------------------------------------------------------------- float64 values

def _norm(x):
    """|x| along the last axis, with the zero subgradient at 0; and where it is not 0."""
    sq = (x * x).sum(-1)
    nz = sq > 0
    return torch.where(nz, torch.where(nz, sq, torch.ones_like(sq)).sqrt(), torch.zeros_like(sq)), nz


def _unit(x):
    n, nz = _norm(x)
    return x / torch.where(nz, n, torch.ones_like(n))[..., None], n, nz


def _cross(a, b):
    a, b = torch.broadcast_tensors(a, b)
    return torch.linalg.cross(a, b, dim=-1)


def _skew(w):
    z = torch.zeros_like(w[..., 0])
    return torch.stack([z, -w[..., 2], w[..., 1], w[..., 2], z, -w[..., 0], -w[..., 1], w[..., 0], z], -1).reshape(w.shape[:-1] + (3, 3))


def _exp(w):
    a2 = (w * w).sum(-1)
    small = a2 < 1e-16
    a = torch.where(small, torch.ones_like(a2), a2).sqrt()
    K = _skew(w)
    c1 = torch.where(small, 1 - a2 / 6, a.sin() / a)
    c2 = torch.where(small, 0.5 - a2 / 24, 2 * (a / 2).sin() ** 2 / (a * a))
    return torch.eye(3, dtype=F64, device=DEV) + c1[..., None, None] * K + c2[..., None, None] * (K @ K)


def _points(h, q):
    """Hand points [B, P, 3] of q [B, D]."""
    t = lambda a: torch.tensor(a, dtype=F64, device=DEV)  # noqa: E731
    T, axis, s, lop = t(h["T_fix"]), t(h["axis"]), t(h["pts"]), torch.tensor(h["lop"], device=DEV, dtype=torch.long)
    R, o = [_exp(q[:, 3:6])], [q[:, :3]]
    for l in range(1, h["L"]):
        p = int(h["parent"][l])
        R.append(R[p] @ T[l, :, :3] @ _exp(q[:, 5 + l, None] * axis[l]))
        o.append(o[p] + R[p] @ T[l, :, 3])
    R, o = torch.stack(R, 1), torch.stack(o, 1)
    return (R[:, lop] @ s[:, :, None])[..., 0] + o[:, lop]


def _grid_lookup(o, p):
    """Trilinear value and gradient at p [..., 3]; outside the grid, at the nearest point of it plus the distance."""
    G = o["grid64"]
    n = torch.tensor([G.shape[2] - 1, G.shape[1] - 1, G.shape[0] - 1], dtype=F64, device=DEV)
    hp = o["pitch"]
    u = (p - torch.tensor(o["origin"], dtype=F64, device=DEV)) / hp
    uc = torch.minimum(u.clamp(min=0), n)
    out = (u < 0) | (u > n)
    i = torch.minimum(uc.detach().floor(), n - 1).long()
    f = uc - i
    du = torch.where(out, u - uc, torch.zeros_like(u))
    eh, e, _ = _unit(du)
    ny, nx = G.shape[1], G.shape[2]
    at = (i[..., 2] * ny + i[..., 1]) * nx + i[..., 0]
    c = [G.reshape(-1)[at + dz * ny * nx + dy * nx + dx] for dz in (0, 1) for dy in (0, 1) for dx in (0, 1)]
    fx, fy, fz = f[..., 0], f[..., 1], f[..., 2]
    lx = [c[2 * k] + fx * (c[2 * k + 1] - c[2 * k]) for k in range(4)]
    dx = [c[2 * k + 1] - c[2 * k] for k in range(4)]
    ly = [lx[0] + fy * (lx[1] - lx[0]), lx[2] + fy * (lx[3] - lx[2])]
    gx = [dx[0] + fy * (dx[1] - dx[0]), dx[2] + fy * (dx[3] - dx[2])]
    dy = [lx[1] - lx[0], lx[3] - lx[2]]
    val = ly[0] + fz * (ly[1] - ly[0])
    g = torch.stack([gx[0] + fz * (gx[1] - gx[0]), dy[0] + fz * (dy[1] - dy[0]), ly[1] - ly[0]], -1) / hp
    return val + hp * e, torch.where(out, torch.zeros_like(g), g) + eh


def _mesh_normals(o):
    if "N" not in o:
        V, F = o["V"].astype(np.float64), o["F"]
        X = V[F]
        fn = np.cross(X[:, 1] - X[:, 0], X[:, 2] - X[:, 0])
        fn /= np.linalg.norm(fn, axis=1, keepdims=True)
        vn = np.zeros_like(V)
        for k in range(3):
            a, b = X[:, (k + 1) % 3] - X[:, k], X[:, (k + 2) % 3] - X[:, k]
            cos = (a * b).sum(1) / np.linalg.norm(a, axis=1) / np.linalg.norm(b, axis=1)
            np.add.at(vn, F[:, k], np.arccos(np.clip(cos, -1, 1))[:, None] * fn)
        t = lambda a: torch.tensor(a, dtype=F64, device=DEV)  # noqa: E731
        o["N"], o["X"] = t((vn / np.linalg.norm(vn, axis=1, keepdims=True))[F]), t(X)
        o["fn"] = t(fn)
    return o["X"], o["N"], o["fn"]


def _mesh_lookup(o, p):
    """Phong distance (blend 3/4) and its gradient; the Phong point is held fixed in the derivative.  The meshes
    here are convex: a point is inside where it is behind every face."""
    X, N, fn = _mesh_normals(o)
    a, ab, ac = X[:, 0], X[:, 1] - X[:, 0], X[:, 2] - X[:, 0]
    d00, d01, d11 = (ab * ab).sum(-1), (ab * ac).sum(-1), (ac * ac).sum(-1)
    den = d00 * d11 - d01 * d01
    flat = p.detach().reshape(-1, 3)
    rho_pt, sign = torch.empty_like(flat), torch.empty_like(flat[:, 0])
    for s in range(0, len(flat), 1 << 16):
        x = flat[s:s + (1 << 16)]
        e1, e2, ea = x @ ab.T - (a * ab).sum(-1), x @ ac.T - (a * ac).sum(-1), x @ a.T
        ap2 = (x * x).sum(-1, keepdim=True) - 2 * ea + (a * a).sum(-1)
        best, bv, bw = None, None, None
        v, w = (d11 * e1 - d01 * e2) / den, (d00 * e2 - d01 * e1) / den
        inside = (v >= 0) & (w >= 0) & (v + w <= 1)
        t_ab, t_ac = (e1 / d00).clamp(0, 1), (e2 / d11).clamp(0, 1)
        t_bc = (((e2 - e1) + d00 - d01) / (d00 + d11 - 2 * d01)).clamp(0, 1)
        for cv, cw, ok in ((v, w, inside), (t_ab, 0 * t_ab, None), (0 * t_ac, t_ac, None), (1 - t_bc, t_bc, None)):
            d2 = ap2 - 2 * (cv * e1 + cw * e2) + cv * cv * d00 + 2 * cv * cw * d01 + cw * cw * d11
            if ok is not None:
                d2 = torch.where(ok, d2, torch.full_like(d2, 1e30))
            if best is None:
                best, bv, bw = d2, cv, cw
            else:
                less = d2 < best
                best, bv, bw = torch.where(less, d2, best), torch.where(less, cv, bv), torch.where(less, cw, bw)
        f = best.argmin(1)
        bv, bw = bv.gather(1, f[:, None]), bw.gather(1, f[:, None])
        bary = torch.cat([1 - bv - bw, bv, bw], 1)
        q = (bary[..., None] * X[f]).sum(1)
        psi = q[:, None] - ((q[:, None] - X[f]) * N[f]).sum(-1, keepdim=True) * N[f]
        rho_pt[s:s + (1 << 16)] = 0.25 * q + 0.75 * (bary[..., None] * psi).sum(1)
        behind = ((x @ fn.T - (a * fn).sum(-1)) < 0).all(1)
        sign[s:s + (1 << 16)] = torch.where(behind, -1.0, 1.0).to(F64)
    sign = sign.reshape(p.shape[:-1])
    u, d, _ = _unit(p - rho_pt.reshape(p.shape))
    return sign * d, sign[..., None] * u


def _lookup(o, p):
    return _mesh_lookup(o, p) if "V" in o else _grid_lookup(o, p)


def _force(o, P, d, n, s, C):
    """Correction of a constraint of value C with lever d, normal n and material displacement s."""
    im, ii = 1.0 / o["mass"], 1.0 / o["inertia"]
    un = _cross(d, n)
    lam_n = C / (im + ii * (un * un).sum(-1))
    t, sig, nz = _unit(s - (s * n).sum(-1, keepdim=True) * n)
    ut = _cross(d, t)
    lam_t = torch.where(nz, torch.where(sig.detach() <= P["mu"] * C.detach(), sig, P["mu"] * C), torch.zeros_like(sig))
    lam_t = lam_t / (im + ii * (ut * ut).sum(-1))
    return -(lam_n[..., None] * n + lam_t[..., None] * t)


def _leaky(phi, P):
    return torch.where(phi.detach() < 0, -phi, -P["alpha_leak"] * (phi - phi.detach()))


def _metric(o, P, p, r, form, T):
    """L_stable + w_pen L_pen [B] of points p [B, P, 3]; and the wrenches."""
    im, ii, dt = 1.0 / o["mass"], 1.0 / o["inertia"], P["dt"]
    V = torch.zeros(M, 3, dtype=F64, device=DEV)
    for m in range(1, M):
        V[m, (m - 1) // 2] = P["v_test"] * (1 if m % 2 else -1)
    B = p.shape[0]
    pe = p[:, :, None]
    if form == "tstep":
        x, w = torch.zeros(B, M, 3, dtype=F64, device=DEV), torch.zeros(B, M, 3, dtype=F64, device=DEV)
        R, v, W, pen = torch.eye(3, dtype=F64, device=DEV).expand(B, M, 3, 3), V.expand(B, M, 3), None, 0.0
        for _ in range(T):
            xt, Rt = x + dt * v, _exp(dt * w) @ R
            d = pe - xt[:, None]
            rr = (d[..., None, :] @ Rt[:, None])[..., 0, :]
            phi, g = _lookup(o, rr)
            n = (Rt[:, None] @ _unit(g)[0][..., None])[..., 0]
            C = _leaky(phi - r, P)
            f = _force(o, P, d, n, pe - x[:, None] - (R[:, None] @ rr[..., None])[..., 0], C)
            N = ((phi.detach() - r) < 0).sum(1).clamp(min=1)[..., None]
            dx, dth = im * f.sum(1) / N, ii * _cross(d, f).sum(1) / N
            x, R, v, w = xt + dx, _exp(dth) @ Rt, (xt + dx - x) / dt, w + dth / dt
        return (_norm(v)[0] + _norm(w)[0]).sum(-1) / M, W
    phi, g = _lookup(o, p)
    n = _unit(g)[0]
    xt = dt * V
    if form == "gs":
        return _sweep(o, P, p, n, phi - r, xt, V), None
    n = n[:, :, None].expand(-1, -1, M, -1)
    phm = (phi - r)[..., None] - (n * xt).sum(-1)
    C, d = _leaky(phm, P), pe - xt
    f = _force(o, P, d, n, xt.expand_as(d), C)
    W = torch.cat([f.sum(1), _cross(d, f).sum(1)], -1)
    N = (phm.detach() < 0).sum(1).clamp(min=1)[..., None]
    L = (_norm(V + im * W[..., :3] / N / dt)[0] + _norm(ii * W[..., 3:] / N / dt)[0]).sum(-1) / M
    return L + P["w_pen"] * C[..., 0].sum(1), W


def _sweep(o, P, p, n, phi_hat, xt, V):
    """The constraints projected one after another in point order; inertia may differ per candidate."""
    im, ii = 1.0 / o["mass"], (1.0 / o["inertia"])
    B = p.shape[0]
    dx, dth, pen = torch.zeros(B, M, 3, dtype=F64, device=DEV), torch.zeros(B, M, 3, dtype=F64, device=DEV), 0.0
    for pi, ni, ph in zip(p.unbind(1), n.unbind(1), phi_hat.unbind(1)):
        ni = ni[:, None].expand(B, M, 3)
        d = pi[:, None] - xt
        D = xt + dx + _cross(dth, d)
        phi = ph[:, None] - (ni * D).sum(-1)
        held = ph[:, None] - (ni * (xt + dx.detach() + _cross(dth.detach(), d))).sum(-1)
        C = torch.where(phi.detach() < 0, -phi, -P["alpha_leak"] * (held - held.detach()))
        f = _force(o, P, d, ni, D, C)
        dx, dth = dx + im * f, dth + (ii[..., None] if torch.is_tensor(ii) else ii) * _cross(d, f)
        pen = pen + C[:, 0]
    return (_norm(V + dx / P["dt"])[0] + _norm(dth / P["dt"])[0]).sum(-1) / M + P["w_pen"] * pen


def _joint_terms(h, P, q):
    lo, hi = (torch.tensor(h[k], dtype=F64, device=DEV) for k in ("q_low", "q_up"))
    th = q[:, 6:]
    return P["w_range"] * _norm(th - 0.5 * (lo + hi))[0] + P["w_limit"] * ((th - hi).clamp(min=0) + (lo - th).clamp(min=0)).sum(-1)


def exact(case, seed):
    form = case["path"] if case["path"] in ("gs", "tstep") else "average"
    rng = np.random.default_rng(seed)
    h = _hand(case["hand"], case["ppl"])
    objs = list(_objects(case, rng))
    q32, oc = _candidates(case, rng, h, np.array([o["rb"] for o in objs]))
    P = {k: float(np.float32(v)) for k, v in _params(case).items() if not isinstance(v, str)}
    r = float(np.float32(_dilation(case)))
    q64 = torch.tensor(q32, dtype=F64, device=DEV)
    per = case["per_obj"]
    if case["path"] == "quality":
        return _exact_quality(case, h, objs, q64, seed)
    if case["path"] == "stages":
        o = _with64(objs[0])
        outs = []
        for s in range(0, per, 64):
            p = _points(h, q64[s:s + 64])
            phi, g = _lookup(o, p)
            outs.append((p, phi - r, g, _metric(o, P, p, r, form, 0)[1]))
        p, phi, g, W = (torch.cat(x) for x in zip(*outs))
        flat = lambda x: x.reshape(-1, 3).T.contiguous()  # noqa: E731
        return {"points": flat(p), "phi": phi.reshape(-1), "phi_grad": flat(g), "wrench": W, "contacts": None, "bits": None}
    if form == "gs" and len(q32) * h["P"] > 2048 * 4352:
        return None
    loss, grad = torch.empty(len(q32), dtype=F64, device=DEV), torch.empty_like(q64)
    if form == "gs":                                    # one sweep over the points for the candidates of all objects
        q = q64.clone().requires_grad_(True)
        p = _points(h, q)
        parts = [_lookup(_with64(o), p[k * per:(k + 1) * per]) for k, o in enumerate(objs)]
        phi, n = torch.cat([x[0] for x in parts]), _unit(torch.cat([x[1] for x in parts]))[0]
        V = torch.zeros(M, 3, dtype=F64, device=DEV)
        for m in range(1, M):
            V[m, (m - 1) // 2] = P["v_test"] * (1 if m % 2 else -1)
        inertia = torch.tensor(np.repeat([o["inertia"] for o in objs], per), dtype=F64, device=DEV)[:, None]
        L = _sweep({"mass": 1.0, "inertia": inertia}, P, p, n, phi - r, P["dt"] * V, V) + _joint_terms(h, P, q)
        (g,) = torch.autograd.grad(L.sum(), q)
        loss, grad = L.detach(), g
    else:
        step = max(1, (1 << 20) // (h["P"] * (8 if form == "tstep" else 1)))
        for k, o in enumerate(objs):
            _with64(o)
            for s in range(k * per, (k + 1) * per, step):
                q = q64[s:min(s + step, (k + 1) * per)].clone().requires_grad_(True)
                L = _metric(o, P, _points(h, q), r, form, case.get("sim_steps", 0))[0] + _joint_terms(h, P, q)
                (g,) = torch.autograd.grad(L.sum(), q)
                loss[s:s + len(q)], grad[s:s + len(q)] = L.detach(), g
            o.pop("grid64", None)
    if case["path"] in ("step", "host"):
        return {"q": q64 - P["lr"] * grad, "loss": loss}
    # A mesh point on the Phong surface has a normal of any direction and a curvature without bound; in the
    # Gauss-Seidel chain every later state hangs on it, so float32 positions give that gradient no digits.
    return {"loss": loss, "grad": None if form == "gs" and case["objects"] == "mesh" else grad}


def _with64(o):
    if "grid" in o and "grid64" not in o:
        o["grid64"] = o["grid"].to(F64)
    return o


def _exact_quality(case, h, objs, q64, seed):
    tau, mu, per = float(np.float32(case["tau"])), float(np.float32(case["mu"])), case["per_obj"]
    area = torch.tensor(h["area"], dtype=F64, device=DEV)
    U = torch.tensor(_directions(case, seed), dtype=F64, device=DEV)
    ang = 2 * math.pi * torch.arange(case["edges"], dtype=F64, device=DEV) / case["edges"]
    eps, ca = [], []
    for k, o in enumerate(objs):
        _with64(o)
        for s in range(k * per, (k + 1) * per, 128):
            p = _points(h, q64[s:min(s + 128, (k + 1) * per)])
            phi, g = _lookup(o, p)
            hit = phi < tau
            ca.append((hit * area).sum(1))
            n = _unit(g)[0]
            sg = torch.where(n[..., 2] >= 0, 1.0, -1.0).to(F64)      # tangent basis of Duff et al. (2017)
            a = -1 / (sg + n[..., 2])
            b = n[..., 0] * n[..., 1] * a
            t1 = torch.stack([1 + sg * n[..., 0] ** 2 * a, sg * b, -sg * n[..., 0]], -1)
            t2 = torch.stack([b, sg + n[..., 1] ** 2 * a, -n[..., 1]], -1)
            for i in range(len(p)):
                at = hit[i].nonzero()[:, 0]
                if not len(at):
                    eps.append(torch.tensor(-math.inf, dtype=F64, device=DEV))
                    continue
                f = -n[i, at, None] + mu * (ang.cos()[:, None] * t1[i, at, None] + ang.sin()[:, None] * t2[i, at, None])
                W = torch.cat([f, 12.5 * _cross(p[i, at, None], f)], -1).reshape(-1, 6)
                eps.append((U @ W.T).max(1).values.min())
        o.pop("grid64", None)
    return {"area": torch.cat(ca), "eps": torch.stack(eps), "contacts": None}
