"""The library's performance cases: what its users run, over the sizes they run it at.

Geometry is what boundary solvers of this kind mesh: geodesic spheres, axis-aligned cubes,
packs of spheres, and forests of such packs.  A case names its task, geometry, kernel and
the plan's knobs; the seed draws the densities, the magnetization or applied field, and,
where the geometry is itself the request's input, its orientation.  Orders and leaf
capacities are the ones the library's workloads and server use: p = 10 for the double
layer, p = 11 for the gradient kernels, and capacities between 32 and 192.
"""
import functools
import math
import random

import numpy as np
import torch

from paper_1605_01715_gb300 import Plan, Tree, capi

PI4 = 4.0 * math.pi
DELTA = 1e-5                    # pairs closer than this contribute nothing
EXACT_PAIRS = 8e10              # direct sums of more pairs take longer than about 20 seconds


def listed():
    return [
        # the smallest request a server sees: one sphere of 2,000 elements, launch latency
        dict(name="sl_sphere_2k", task="matvec", call="direct", shape="sphere", size=10, bodies=1, kernel="sl", p=6,
             leaf=64, precision="mixed", cut=0.0),
        # the everyday single-layer sum (20,480 elements)
        dict(name="sl_sphere_20k", task="matvec", call="direct", shape="sphere", size=32, bodies=1, kernel="sl", p=6,
             leaf=64, precision="mixed", cut=0.0),
        # the demagnetization matvec of a cube inside a long solve: replayed, on the device
        dict(name="demag_cube_1m", task="matvec", call="graph", shape="cube", size=296, bodies=1, kernel="dl", p=10,
             leaf=192, precision="mixed", cut=1e-8),
        # the same for a caller whose densities live in pinned host memory (270,000 elements)
        dict(name="demag_cube_270k_host", task="matvec", call="host", shape="cube", size=150, bodies=1, kernel="dl",
             p=10, leaf=192, precision="mixed", cut=0.0),
        # one demagnetizing potential of a large curved body
        dict(name="demag_sphere_1m", task="demag", call="direct", shape="sphere", size=229, bodies=1, kernel="dl",
             p=10, leaf=128, precision="mixed", cut=0.0),
        # one application of the polarization operator of a 64-body suspension (677,120 unknowns)
        dict(name="polar_64_apply", task="apply", call="direct", shape="pack", size=23, bodies=64, kernel="adl", p=11,
             leaf=96, precision="mixed", cut=0.0),
        # a whole polarization solve of a small suspension
        dict(name="polar_8_solve", task="solve", call="direct", shape="pack", size=10, bodies=8, kernel="adl", p=11,
             leaf=96, precision="mixed", cut=0.0),
        # the field at the elements after such a solve, on the solve's tree
        dict(name="field_pack_32", task="field", call="direct", shape="pack", size=17, bodies=32, kernel="field", p=11,
             leaf=96, precision="mixed", cut=0.0),
        # many uneven instances in one forest
        dict(name="batch_24", task="matvec", call="graph", shape="forest", size=30000, bodies=24, kernel="sl", p=8,
             leaf=64, precision="mixed", cut=0.0),
        # the interior field of a magnetized sphere at a ragged number of volume targets
        dict(name="interior_5001", task="targets", call="direct", shape="sphere", size=101, bodies=5001, kernel="adl",
             p=11, leaf=128, precision="mixed", cut=0.0),
        # the FP64 form, as the reference the orders are tuned against
        dict(name="fp64_sphere_46k", task="matvec", call="direct", shape="sphere", size=48, bodies=1, kernel="sl",
             p=12, leaf=64, precision="fp64", cut=0.0),
        # one request from triangles to potential: quadrature, tree, plan, matvec
        dict(name="request_sphere_98k", task="request", call="direct", shape="sphere", size=70, bodies=1, kernel="dl",
             p=10, leaf=96, precision="mixed", cut=0.0),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    task = rng.choice(["matvec", "matvec", "demag", "apply", "solve", "field", "forest", "targets", "fp64", "request"])
    leaf = rng.choice([48, 64, 96, 128, 160, 192])
    case = dict(task=task, call="direct", shape="sphere", size=0, bodies=1, kernel="sl", p=6, leaf=leaf,
                precision="mixed", cut=0.0)
    if task == "matvec":
        case["call"] = rng.choice(["direct", "graph", "host"])
        case["kernel"] = rng.choice(["sl", "dl"])
        case["shape"] = rng.choice(["sphere", "cube"])
        case["p"] = rng.choice([6, 8, 10]) if case["kernel"] == "sl" else 10
        case["size"] = _log_int(rng, 10, 180) if case["shape"] == "sphere" else _log_int(rng, 13, 250)
        if case["shape"] == "cube" and case["kernel"] == "dl":
            case["cut"] = rng.choice([0.0, 1e-8])
    elif task == "demag":
        case.update(kernel="dl", p=10, size=_log_int(rng, 12, 200), shape=rng.choice(["sphere", "cube"]))
    elif task == "apply":
        bodies = _log_int(rng, 1, 64)
        case.update(kernel="adl", p=11, shape="pack", bodies=bodies, size=_log_int(rng, 7, 23))
    elif task == "solve":
        bodies = _log_int(rng, 1, 12)
        case.update(kernel="adl", p=11, shape="pack", bodies=bodies, size=_log_int(rng, 6, 12))
    elif task == "field":
        case.update(kernel="field", p=11, shape="pack", bodies=_log_int(rng, 1, 32), size=_log_int(rng, 8, 17))
    elif task == "forest":
        case.update(task="matvec", call=rng.choice(["direct", "graph"]), shape="forest", p=8,
                    bodies=_log_int(rng, 3, 24), size=_log_int(rng, 3000, 30000))
    elif task == "targets":
        case.update(kernel=rng.choice(["adl", "sl", "dl"]), bodies=_log_int(rng, 300, 40000),
                    size=_log_int(rng, 20, 101))
        case["p"] = 11 if case["kernel"] == "adl" else 10
    elif task == "fp64":
        case.update(task="matvec", kernel=rng.choice(["sl", "dl"]), precision=rng.choice(["fp64", "fp64", "cheb_fp64"]),
                    size=_log_int(rng, 10, 40))
        case["p"] = rng.choice([5, 6]) if case["precision"] == "cheb_fp64" else rng.choice([10, 11, 12])
        case["leaf"] = rng.choice([40, 64, 96])
    else:
        case.update(kernel="dl", p=10, shape=rng.choice(["sphere", "cube"]), size=_log_int(rng, 12, 70),
                    leaf=rng.choice([64, 96, 128]))
    return case


# ---------------------------------------------------------------- geometry (triangle soups)
def _sphere_soup(freq):
    """Unit geodesic sphere: every icosahedron face cut into freq^2 triangles, pushed out."""
    g = (1.0 + math.sqrt(5.0)) / 2.0
    verts = []
    for a in (-1.0, 1.0):
        for b in (-g, g):
            verts += [(0.0, a, b), (a, b, 0.0), (b, 0.0, a)]
    v = np.array(verts)
    faces = []
    for i in range(12):
        for j in range(i + 1, 12):
            for k in range(j + 1, 12):
                if max(np.sum((v[i] - v[j]) ** 2), np.sum((v[j] - v[k]) ** 2), np.sum((v[i] - v[k]) ** 2)) < 4.1:
                    outward = np.linalg.det(v[[i, j, k]]) > 0
                    faces.append((i, j, k) if outward else (i, k, j))
    v /= np.linalg.norm(v, axis=1, keepdims=True)
    i, j = np.meshgrid(np.arange(freq), np.arange(freq), indexing="ij")
    i, j = i.ravel(), j.ravel()
    up, dn = i + j < freq, i + j < freq - 1
    cells = [[(i[up], j[up]), (i[up] + 1, j[up]), (i[up], j[up] + 1)],
             [(i[dn] + 1, j[dn]), (i[dn] + 1, j[dn] + 1), (i[dn], j[dn] + 1)]]
    out = []
    for f in faces:
        for cell in cells:
            tri = [((freq - ci - cj)[:, None] * v[f[0]] + ci[:, None] * v[f[1]] + cj[:, None] * v[f[2]]) / freq
                   for ci, cj in cell]
            out.append(np.stack(tri, axis=1))
    tri = np.concatenate(out)
    return tri / np.linalg.norm(tri, axis=2, keepdims=True)


def _cube_soup(n):
    """Unit cube around the origin, n x n squares of two triangles on each face."""
    u, w = np.meshgrid(np.arange(n), np.arange(n), indexing="ij")
    grid = np.linspace(-0.5, 0.5, n + 1)
    out = []
    for axis in range(3):
        for side in (0.5, -0.5):
            b, c = (axis + 1) % 3, (axis + 2) % 3
            if side < 0:
                b, c = c, b

            def corner(du, dw):
                p = np.empty((n * n, 3))
                p[:, axis] = side
                p[:, b] = grid[(u + du).ravel()]
                p[:, c] = grid[(w + dw).ravel()]
                return p

            p00, p10, p11, p01 = corner(0, 0), corner(1, 0), corner(1, 1), corner(0, 1)
            out += [np.stack([p00, p10, p11], 1), np.stack([p00, p11, p01], 1)]
    return np.concatenate(out)


def _pack(bodies, seed):
    """Centres and radii (0.5 to 1.5) of spheres with surface gaps of 0.05 or more, at the
    density of 64 spheres in a box of edge 20."""
    rng = random.Random(seed)
    box = max(4.0, 20.0 * (bodies / 64.0) ** (1.0 / 3.0))
    while True:
        c, r = [], []
        for _ in range(bodies):
            ri = rng.uniform(0.5, 1.5)
            for _ in range(2000):
                x = [rng.uniform(ri, box - ri) for _ in range(3)]
                if all(math.dist(x, y) >= ri + s + 0.05 for y, s in zip(c, r)):
                    c.append(x)
                    r.append(ri)
                    break
        if len(c) == bodies:
            return np.array(c), np.array(r)
        box *= 1.05


@functools.lru_cache(maxsize=6)
def _mesh(shape, size, bodies):
    """(tri (T, 3, 3), sph (T, 4), body (T,), instance offsets or None) on the host."""
    if shape == "cube":
        tri = _cube_soup(size)
        return tri, np.zeros((len(tri), 4)), np.zeros(len(tri), np.int32), None
    if shape == "sphere":
        tri = _sphere_soup(size)
        sph = np.tile(np.array([0.0, 0.0, 0.0, 1.0]), (len(tri), 1))
        return tri, sph, np.zeros(len(tri), np.int32), None
    if shape == "pack":
        c, r = _pack(bodies, 3000 + bodies)
        unit = _sphere_soup(size)
        tri = np.concatenate([unit * ri + ci for ci, ri in zip(c, r)])
        sph = np.repeat(np.concatenate([c, r[:, None]], 1), len(unit), axis=0)
        return tri, sph, np.repeat(np.arange(bodies, dtype=np.int32), len(unit)), None
    # forest: `bodies` packs of 1 to 24 spheres, sizes log-uniform from 1,000 elements to `size`
    rng = random.Random(4000 + bodies)
    tris, sphs, off = [], [], [0]
    for i in range(bodies):
        want = math.exp(rng.uniform(math.log(1000), math.log(size)))
        ns = rng.randint(1, 24)
        unit = _sphere_soup(max(2, round(math.sqrt(want / (20.0 * ns)))))
        c, r = _pack(ns, 5000 + i)
        tris += [unit * ri + ci for ci, ri in zip(c, r)]
        sphs += [np.tile(np.append(ci, ri), (len(unit), 1)) for ci, ri in zip(c, r)]
        off.append(off[-1] + ns * len(unit))
    return np.concatenate(tris), np.concatenate(sphs), None, tuple(off)


def _soup(case, seed):
    """The case's triangles on the device; a request's sphere is turned by the seed."""
    tri, sph, body, off = _mesh(case["shape"], case["size"], 1 if case["task"] == "targets" else case["bodies"])
    tri_d, sph_d = torch.from_numpy(tri).cuda(), torch.from_numpy(sph).cuda()
    if case["task"] == "request" and case["shape"] == "sphere":
        turn, _ = np.linalg.qr(np.random.default_rng(seed + 77).normal(size=(3, 3)))
        if np.linalg.det(turn) < 0:
            turn[:, 0] = -turn[:, 0]
        tri_d = (tri_d @ torch.from_numpy(turn).cuda().T).contiguous()
    return tri_d, sph_d, body, off


def _points(tri, sph):
    """Centroid, weight and normal of each triangle, (3, T), (T,), (3, T): radial and
    spherical on a sphere, flat otherwise."""
    c = tri.mean(1)
    a, b, d = tri[:, 0], tri[:, 1], tri[:, 2]
    flat = torch.linalg.cross(b - a, d - a)
    area = 0.5 * flat.norm(dim=1)
    nrm = flat / flat.norm(dim=1, keepdim=True)
    on = sph[:, 3] > 0
    rad = sph[:, 3:4].clamp(min=1e-300)
    ua, ub, ud = (x - sph[:, :3] for x in (a, b, d))
    ua, ub, ud = ua / rad, ub / rad, ud / rad
    trip = (ua * torch.linalg.cross(ub, ud)).sum(1).abs()
    den = 1.0 + (ua * ub).sum(1) + (ub * ud).sum(1) + (ud * ua).sum(1)
    curved = 2.0 * torch.atan2(trip, den) * sph[:, 3] ** 2
    out = c - sph[:, :3]
    area = torch.where(on, curved, area)
    nrm = torch.where(on[:, None], out / out.norm(dim=1, keepdim=True), nrm)
    return c.T.contiguous(), area, nrm.T.contiguous()


# ---------------------------------------------------------------- inputs from the seed
def _inputs(case, seed, xyz, w, nrm, body):
    """The task's densities and coefficients on the device, from the seed alone."""
    rng = np.random.default_rng(seed)
    n = w.numel()
    d = rng.normal(size=3)
    d /= np.linalg.norm(d)                      # magnetization or applied field, a unit vector
    dir_d = torch.from_numpy(d).cuda()[:, None]
    got = dict(direction=tuple(float(v) for v in d))
    task = case["task"]
    if task in ("matvec", "targets"):
        if case["kernel"] == "sl":
            sigma = torch.from_numpy(rng.uniform(-1.0, 1.0, n)).cuda()
        else:
            sigma = (dir_d * nrm).sum(0)        # the magnetic surface charge n . M
        got["q"] = sigma * w
    elif task in ("demag", "request"):
        got["phi1"] = PI4 * (dir_d * xyz).sum(0)
        got["omega"] = torch.full_like(w, 2.0 * math.pi)
    elif task in ("apply", "solve", "field"):
        idx = torch.from_numpy(body.astype(np.int64)).cuda()
        got["eps_in"] = torch.from_numpy(rng.uniform(2.0, 20.0, case["bodies"])).cuda()[idx]
        # a charge of the shape a uniform field induces, uneven from body to body
        got["sigma"] = (dir_d * nrm).sum(0) * torch.from_numpy(rng.uniform(0.5, 2.5, case["bodies"])).cuda()[idx]
    if task == "targets":
        # ragged volume targets inside the sphere, each with the unit normal of the wanted component
        m = case["bodies"]
        x = rng.normal(size=(3, m))
        x *= 0.8 * rng.uniform(0.0, 1.0, m) ** (1.0 / 3.0) / np.linalg.norm(x, axis=0)
        got["trg"] = torch.from_numpy(np.ascontiguousarray(x)).cuda()
        got["tnrm"] = dir_d.expand(3, m).contiguous()
    return got


_anchors = {}


def _keep_tables(kernel, p, precision, cut):
    """A small plan of these knobs that stays alive, as a server keeps one, so that the
    operator tables are built once and not by every plan."""
    key = (kernel, p, precision, cut)
    if key not in _anchors:
        xyz, _, nrm = capi.kifmm_quadrature_points(*(torch.from_numpy(a).cuda() for a in _mesh("sphere", 3, 1)[:2]))
        _anchors[key] = Plan(Tree(xyz, max_leaf=64), kernel=kernel, p=p, precision=precision, pinv_cutoff=cut,
                             src_nrm=nrm, trg_nrm=nrm)


def prepare(case, seed):
    _keep_tables(case["kernel"], case["p"], case["precision"], case["cut"])
    tri, sph, body, off = _soup(case, seed)
    xyz, w, nrm = capi.kifmm_quadrature_points(tri, sph)
    st = dict(case=case, **_inputs(case, seed, xyz, w, nrm, body))
    if case["task"] == "request":
        st.update(tri=tri, sph=sph)
        return st
    if case["task"] == "targets":
        tree = Tree(xyz, st["trg"], max_leaf=case["leaf"])
        tnrm = st["tnrm"]
    else:
        tree = Tree(xyz, max_leaf=case["leaf"], instances=off)
        tnrm = nrm
    st["plan"] = Plan(tree, kernel=case["kernel"], p=case["p"], precision=case["precision"], pinv_cutoff=case["cut"],
                      src_nrm=nrm, trg_nrm=tnrm)
    st.update(w=w, nrm=nrm)
    if case["call"] == "graph":
        st["out"] = torch.empty(st["plan"].n_out, dtype=torch.float64, device="cuda")
    elif case["call"] == "host":
        st["q"] = st["q"].cpu().pin_memory()
        st["out"] = torch.empty(st["plan"].n_out, dtype=torch.float64).pin_memory()
    if case["task"] in ("apply", "solve", "field"):
        st["curv"] = 1.0 / sph[:, 3].contiguous()
        st["b"] = capi.kifmm_polarization_rhs(nrm, st["eps_in"], 1.0, st["direction"])
    return st


def run(state):
    case, task = state["case"], state["case"]["task"]
    if task == "request":
        xyz, w, nrm = capi.kifmm_quadrature_points(state["tri"], state["sph"])
        tree = Tree(xyz, max_leaf=case["leaf"])
        plan = Plan(tree, kernel="dl", p=case["p"], precision=case["precision"], pinv_cutoff=case["cut"], src_nrm=nrm)
        return plan.demag_phi2(state["phi1"], w, state["omega"])
    plan = state["plan"]
    if task == "demag":
        return plan.demag_phi2(state["phi1"], state["w"], state["omega"])
    if task == "apply":
        return plan.bie_apply(state["w"], state["eps_in"], 1.0, state["curv"], state["sigma"])
    if task == "solve":
        x, iters, _, _ = plan.bie_solve(state["w"], state["eps_in"], 1.0, state["curv"], state["b"], tol=1e-6,
                                        restart=50, max_iter=500)
        return dict(x=x, iters=iters)
    if task == "field":
        return plan.polarization_field(state["w"], state["curv"], state["nrm"], state["sigma"], state["direction"])
    if case["call"] == "graph":
        return plan.matvec_graph(state["q"], state["out"])
    if case["call"] == "host":
        return plan.matvec_host(state["q"], state["out"])
    return plan.matvec(state["q"])


# ---------------------------------------------------------------- the same in 64 bits, term by term
def _direct(kernel, trg, src, q, snrm, tnrm):
    """Sum over all pairs in FP64, a block of targets at a time."""
    nt, ns = trg.shape[1], src.shape[1]
    out = torch.empty((3, nt) if kernel == "field" else nt, dtype=torch.float64, device="cuda")
    step = max(1, int(1.5e8) // ns)
    for t0 in range(0, nt, step):
        t1 = min(nt, t0 + step)
        d = [trg[k, t0:t1, None] - src[k][None, :] for k in range(3)]
        r2 = d[0] * d[0]
        r2.addcmul_(d[1], d[1]).addcmul_(d[2], d[2])
        inv = r2.rsqrt().masked_fill_(r2 < DELTA * DELTA, 0.0)
        if kernel == "sl":
            out[t0:t1] = inv @ q
            continue
        inv = inv * inv * inv
        if kernel == "field":
            for k in range(3):
                out[k, t0:t1] = (d[k] * inv) @ q
        elif kernel == "adl":
            dot = d[0] * tnrm[0, t0:t1, None]
            dot.addcmul_(d[1], tnrm[1, t0:t1, None]).addcmul_(d[2], tnrm[2, t0:t1, None])
            out[t0:t1] = (dot * inv) @ q
        else:
            dot = d[0] * snrm[0][None, :]
            dot.addcmul_(d[1], snrm[1][None, :]).addcmul_(d[2], snrm[2][None, :])
            out[t0:t1] = (dot * inv) @ q
    return out


def exact(case, seed):
    tri, sph, body, off = _soup(case, seed)
    n = tri.shape[0]
    nt = case["bodies"] if case["task"] == "targets" else n
    pairs = sum((b - a) ** 2 for a, b in zip(off, off[1:])) if off else float(n) * nt
    if pairs > EXACT_PAIRS:
        return None
    xyz, w, nrm = _points(tri, sph)
    st = _inputs(case, seed, xyz, w, nrm, body)
    task, kernel = case["task"], case["kernel"]
    if task in ("demag", "request"):
        dl = _direct("dl", xyz, xyz, st["phi1"] * w, nrm, None)
        return dl / PI4 + (st["omega"] / PI4 - 1.0) * st["phi1"]
    if task in ("apply", "solve", "field"):
        self_term = torch.sqrt(math.pi * w) / sph[:, 3]
        e0 = torch.tensor(st["direction"], dtype=torch.float64, device="cuda")[:, None]
        if task == "field":
            f = _direct("field", xyz, xyz, st["sigma"] * w, None, None)
            return e0 + (f + self_term * st["sigma"] * nrm) / PI4
        mean, jump = 0.5 * (st["eps_in"] + 1.0), 1.0 - st["eps_in"]
        if task == "apply":
            f = _direct("adl", xyz, xyz, st["sigma"] * w, None, nrm)
            return mean * st["sigma"] + jump * (f + self_term * st["sigma"]) / PI4
        if n > 20000:
            return None
        A = torch.empty((n, n), dtype=torch.float64, device="cuda")
        for t0 in range(0, n, 2048):
            t1 = min(n, t0 + 2048)
            d = [xyz[k, t0:t1, None] - xyz[k][None, :] for k in range(3)]
            r2 = d[0] * d[0] + d[1] * d[1] + d[2] * d[2]
            inv = r2.rsqrt().masked_fill_(r2 < DELTA * DELTA, 0.0)
            dot = d[0] * nrm[0, t0:t1, None] + d[1] * nrm[1, t0:t1, None] + d[2] * nrm[2, t0:t1, None]
            A[t0:t1] = jump[t0:t1, None] / PI4 * dot * inv * inv * inv * w[None, :]
        A.diagonal().add_(mean + jump * self_term / PI4)
        b = -jump * (e0 * nrm).sum(0)
        return dict(x=torch.linalg.solve(A, b), iters=None)
    if task == "targets":
        return _direct(kernel, st["trg"], xyz, st["q"], nrm, st["tnrm"])
    if off:
        return torch.cat([_direct(kernel, xyz[:, a:b].contiguous(), xyz[:, a:b].contiguous(), st["q"][a:b], None, None)
                          for a, b in zip(off, off[1:])])
    return _direct(kernel, xyz, xyz, st["q"], nrm, nrm)


# ---------------------------------------------------------------- what a pass cannot do without
def work(case):
    """Bytes: points, normals and densities in, results out, each once.  Flops: the near
    sums over a surface's neighbouring leaves and the translations between projections of
    half the surface points, for a tree of half-full leaves."""
    size, p = case["size"], case["p"]
    if case["shape"] == "cube":
        n = 12 * size * size
    elif case["shape"] == "forest":
        n = case["bodies"] * 0.3 * size
    else:
        n = 20 * size * size * (case["bodies"] if case["shape"] == "pack" else 1)
    nt = case["bodies"] if case["task"] == "targets" else n
    comps = 3 if case["kernel"] == "field" else 1
    pts = 24.0 * n + (24.0 * nt if case["task"] == "targets" else 0.0)
    nrm = 0.0 if case["kernel"] in ("sl", "field") else 24.0 * (nt if case["kernel"] == "adl" else n)
    nbytes = pts + nrm + 8.0 * n + 8.0 * comps * nt
    q = p ** 3 if case["precision"].startswith("cheb") else 6 * (p - 1) ** 2 + 2
    rank = q if case["precision"].startswith("cheb") else 0.5 * q
    pair = {"sl": 10.0, "dl": 18.0, "adl": 18.0, "field": 17.0}[case["kernel"]]
    boxes = 4.0 / 3.0 * n / (0.5 * case["leaf"])
    flops = nt * 6.0 * case["leaf"] * pair + boxes * 27.0 * 2.0 * rank * rank + n * pair * rank + 2.0 * comps * nt * rank
    if case["task"] == "solve":
        flops *= 12.0                               # applications of the operator in a solve
    elif case["task"] == "request":
        nbytes += 104.0 * n                         # the triangles and their spheres
        flops += nt * 2.0 * q * rank                # the targets' evaluation rows
    return {"bytes": nbytes, "flops": flops}
