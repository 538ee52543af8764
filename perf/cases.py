"""The work that users of the library have it do, as measurable cases.

Every case goes through the public entry points (``srp.Context`` and
``autograd``): single evaluations as an outside integrator asks for them,
tables of directions, recorded hits, diffuse rays, gradients, propagated arcs
one by one, in batches and with an interpolated force, and the arc adjoint.
Meshes are the generators' spacecraft of 16 to 200k triangles, ray grids have
64 to 1024 rays a side and 0 to 2 bounces: the ranges of the benchmark, the
tests and the batched workload.  ``exact`` is a brute-force ray tracer in
64-bit torch.
"""
from __future__ import annotations

import functools
import math
from types import SimpleNamespace

import numpy as np
import torch

from paper_2608_07307_gb300 import autograd, inputs, srp

P0 = 4.56e-6
GEO = 42164e3
MU_EARTH, MU_SUN, AU = 3.986004418e14, 1.32712440018e20, 1.495978707e11


def listed():
    return [
        # one Sun direction on the smallest spacecraft: what an outside integrator asks for at each of its stages
        dict(name="boxwing_single", kind="eval", mesh="box_wing", N=256, bounces=1, n=1, dist=True),
        # the box-wing at 256 directions in one call: the plain evaluation workload
        dict(name="boxwing_table", kind="eval", mesh="box_wing", N=256, bounces=1, n=256),
        # one evaluation of a 50k-triangle craft given its attitude: an attitude and orbit simulator's step
        dict(name="craft50k_attitude", kind="eval", mesh="spacecraft", facet=0.05, N=512, bounces=1, n=1, quat=True,
             dist=True, mode="offset"),
        # the headline batch: 200k triangles, 1024^2 rays, two bounces, 32 directions
        dict(name="craft200k_batch", kind="eval", mesh="spacecraft", facet=0.025, N=1024, bounces=2, n=32),
        # a part of a force table at an odd grid and an odd number of directions, joints commanded
        dict(name="craft100k_odd", kind="eval", mesh="spacecraft", facet=0.035, N=777, bounces=2, n=37, mode="set"),
        # hit triangles recorded per ray: visibility studies and validation
        dict(name="craft12k_hits", kind="eval", mesh="spacecraft", facet=0.1, N=301, bounces=2, n=7, hits=True),
        # the paper's ray-trace configuration: 256^2 rays, 16 diffuse rays a hit
        dict(name="craft50k_diffuse", kind="eval", mesh="spacecraft", facet=0.05, N=256, bounces=1, n=8, diffuse=16),
        # forward and backward of the inertial acceleration: estimation of coefficients, joints and attitude
        dict(name="craft50k_grad", kind="grad", mesh="spacecraft", facet=0.05, N=512, bounces=1, n=6),
        # six hours of the GEO arc with the ray-traced force in every stage of RKF7(8)
        dict(name="geo_arc", kind="arc", mesh="spacecraft", facet=0.025, N=512, bounces=1, hours=6.0, n=1),
        # the arc adjoint: half an hour of RK4 at 60 s with checkpoints
        dict(name="geo_adjoint", kind="adjoint", mesh="spacecraft", facet=0.05, N=512, bounces=1, steps=30, every=10),
        # different trajectories, meshes, grids and bounces in one call
        dict(name="arcs_batched", kind="batch", n=24, hours=1.0, facets=4),
        # dispersed arcs on a force table: Monte Carlo runs
        dict(name="arcs_table", kind="table_arcs", mesh="spacecraft", facet=0.1, N=256, bounces=1, n=512, hours=24.0),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["eval"] * 5 + ["diffuse", "grad", "grad", "arc", "adjoint", "batch", "table_arcs"])
    mesh = rng.choice(["box_wing", "box_wing_two_axis", "spacecraft", "spacecraft", "spacecraft", "spacecraft"])
    c = dict(kind=kind, mesh=mesh)
    if mesh == "spacecraft":
        c["facet"] = round(_log(rng, 0.025, 0.4), 4)
    if kind == "batch":
        return dict(kind=kind, n=int(_log(rng, 4, 24)), hours=round(rng.uniform(0.3, 1.0), 2), facets=rng.randint(1, 4))
    c.update(N=int(_log(rng, 64, 1024)), bounces=rng.randint(0, 2))
    if kind == "eval":
        c.update(n=int(_log(rng, 1, min(256, 2 ** 25 // c["N"] ** 2))), mode=rng.choice(["track", "offset", "set"]))
        for key in ("dist", "quat"):
            c[key] = rng.random() < 0.5
        if c["n"] * c["N"] ** 2 < 2 ** 21:
            c["hits"] = rng.random() < 0.3
        return c
    if kind == "diffuse":
        c.update(kind="eval", N=int(_log(rng, 64, 256)), bounces=rng.randint(1, 2), n=int(_log(rng, 1, 16)),
                 diffuse=rng.randint(1, 16))
        return c
    if kind == "table_arcs":
        c.update(N=min(c["N"], 256), n=int(_log(rng, 1, 512)), hours=round(_log(rng, 2, 24), 2))
        return c
    c["bounces"] = rng.randint(0, 1)
    if kind == "grad":
        c.update(N=min(c["N"], 512), n=int(_log(rng, 1, 8)))
    elif kind == "arc":
        c.update(N=min(c["N"], 512), n=rng.choice([1, 1, 2, 3]), hours=round(rng.uniform(1.0, 6.0) / 2, 2))
    else:
        c.update(N=min(c["N"], 512), steps=rng.randint(5, 30), every=rng.randint(3, 12))
    return c


# ---------------------------------------------------------------- preparation
@functools.lru_cache(maxsize=12)
def _geometry(mesh, facet=None):
    if mesh == "spacecraft":
        return inputs.spacecraft(facet)
    return inputs.box_wing() if mesh == "box_wing" else inputs.box_wing_two_axis()


def _mesh(case, rng):
    """The case's spacecraft, its optical coefficients drawn anew."""
    m = _geometry(case["mesh"], case.get("facet"))
    return m.with_materials(rng.uniform(0.0, 0.5, (len(m.mat), 2)))


def _sphere(rng, n):
    z, phi = rng.uniform(-1.0, 1.0, n), rng.uniform(0.0, 2.0 * math.pi, n)
    r = np.sqrt(1.0 - z * z)
    return np.stack([r * np.cos(phi), r * np.sin(phi), z], axis=1)


def _quats(rng, n):
    q = rng.normal(size=(n, 4))
    return q / np.linalg.norm(q, axis=1, keepdims=True)


def _joints(m, mode, rng):
    a = np.zeros(len(m.parent))
    movable = np.abs(m.axis).sum(axis=1) > 0
    movable[0] = False
    if mode != "track":
        a[movable] = rng.uniform(-1.0, 1.0, movable.sum()) * (0.1 if mode == "offset" else 0.5)
    return a


MODES = {"track": srp.PANELS_TRACK, "offset": srp.PANELS_TRACK_OFFSET, "set": srp.PANELS_SET}


def _arrays(case, seed):
    """The inputs of an evaluation or its gradient, in numpy."""
    rng = np.random.default_rng([seed, 1])
    v = SimpleNamespace(mesh=_mesh(case, rng), mode=case.get("mode", "track"))
    n = case["n"]
    v.dirs = _sphere(rng, n)
    v.dist = rng.uniform(0.7, 1.2, n)
    v.quat = _quats(rng, n)
    v.angles = _joints(v.mesh, v.mode, rng)
    v.seed = int(rng.integers(1 << 31))
    v.g_acc, v.g_torque = rng.normal(size=(n, 3)), rng.normal(size=(n, 3))
    return v


def _geo_state(rng):
    ph, inc = rng.uniform(0.0, 2.0 * math.pi), math.radians(0.1)
    v = math.sqrt(MU_EARTH / GEO)
    y = np.array([GEO * math.cos(ph), GEO * math.sin(ph), 0.0, -v * math.sin(ph) * math.cos(inc),
                  v * math.cos(ph) * math.cos(inc), v * math.sin(inc)])
    return y + np.concatenate([rng.normal(scale=1e3, size=3), rng.normal(scale=1.0, size=3)])


def prepare(case, seed):
    st = SimpleNamespace(case=case, stream=torch.cuda.Stream())
    st.ctx = srp.Context(0, st.stream)
    kind = case["kind"]
    gpu = functools.partial(torch.tensor, dtype=torch.float64, device="cuda:0")
    rng = np.random.default_rng([seed, 2])
    if kind in ("eval", "grad"):
        v = _arrays(case if kind == "eval" else dict(case, mode="offset"), seed)
        st.mid = st.ctx.load_mesh(v.mesh)
        st.dirs, st.dist, st.quat = gpu(v.dirs), gpu(v.dist), gpu(v.quat)
        if kind == "grad":
            st.mat, st.angles = gpu(v.mesh.mat), gpu(v.angles)
            st.g_acc, st.g_torque = gpu(v.g_acc), gpu(v.g_torque)
        else:
            st.ctx.set_panel_angles(st.mid, v.angles)
            st.opts = dict(N=case["N"], bounces=case["bounces"], panel_mode=MODES[v.mode], hits=bool(case.get("hits")),
                           n_diffuse=case.get("diffuse", 0), diffuse_seed=v.seed)
    elif kind in ("arc", "adjoint", "table_arcs"):
        st.mid = st.ctx.load_mesh(_mesh(case, rng))
        n = case.get("n", 1)
        st.y0 = np.stack([_geo_state(rng) for _ in range(n)])
        if kind == "adjoint":
            st.t01, st.g_y1 = np.array([[0.0, 60.0 * case["steps"]]]), rng.normal(size=(1, 6))
        else:
            st.t01 = np.tile([[0.0, 3600.0 * case["hours"]]], (n, 1))
        if kind == "table_arcs":
            st.table = st.ctx.spad_build(st.mid, inputs.SPAD_20x10, N=case["N"], bounces=case["bounces"], device=True)
    else:
        facets = [0.4, 0.2, 0.1, 0.05][: case["facets"]]
        meshes = [_mesh(dict(mesh="spacecraft", facet=f), rng) for f in facets]
        mids = [st.ctx.load_mesh(m) for m in meshes]
        st.trajs = []
        for k in range(case["n"]):
            mi, mode = k % len(mids), ["track", "offset", "set"][int(rng.integers(3))]
            # the same spread of grids, bounces and orbits for every seed, so that one size means one amount of work
            t = dict(mesh_id=mids[mi], N=[256, 512, 333, 768][(k // 2) % 4], bounces=k % 3, panel_mode=MODES[mode],
                     angles=_joints(meshes[mi], mode, rng) if mode != "track" else None, q=tuple(_quats(rng, 1)[0]), t0=0.0)
            if k % 2 == 0:
                t.update(central=0, attitude=0, y0=_geo_state(rng), t1=3600.0 * case["hours"])
            else:
                r, ph = rng.uniform(0.7, 1.2) * AU, rng.uniform(0.0, 2.0 * math.pi)
                s = math.sqrt(MU_SUN / r)
                t.update(central=1, attitude=1, t1=2.0 * 86400.0 * case["hours"],
                         y0=np.array([r * math.cos(ph), r * math.sin(ph), 0.0, -s * math.sin(ph), s * math.cos(ph), 0.0]))
            st.trajs.append(t)
    torch.cuda.synchronize()
    return st


# ----------------------------------------------------------------------- runs
def run(st):
    case, ctx = st.case, st.ctx
    kind = case["kind"]
    with torch.cuda.stream(st.stream):
        if kind == "eval":
            out = ctx.eval_batch(st.mid, st.dirs, sun_dist=st.dist if case.get("dist") else None,
                                 quat=st.quat if case.get("quat") else None, **st.opts)
            return dict(zip(("force", "torque", "hits"), out))
        if kind == "grad":
            leaf = [x.detach().requires_grad_(True) for x in (st.quat, st.dirs, st.dist, st.mat, st.angles)]
            acc, torque = autograd.srp_accel_inertial(ctx, st.mid, *leaf, N=case["N"], bounces=case["bounces"])
            torch.autograd.backward([acc, torque], [st.g_acc, st.g_torque])
            names = ("g_quat", "g_sun", "g_dist", "g_mat", "g_angles")
            return dict(zip(names, [x.grad for x in leaf]), acc=acc.detach(), torque=torque.detach())
        kw = dict(j2=True, sun3=True)
        if kind == "arc":
            y1, _, _ = ctx.propagate(st.mid, st.y0, st.t01, N=case["N"], bounces=case["bounces"], **kw)
            return y1
        if kind == "table_arcs":
            y1, _, _ = ctx.propagate(st.mid, st.y0, st.t01, spad=(inputs.SPAD_20x10, st.table), **kw)
            return y1
        if kind == "adjoint":
            g = ctx.prop_grad(st.mid, st.y0, st.t01, st.g_y1, ckpt_every=case["every"], N=case["N"],
                              bounces=case["bounces"], **kw)
            return {k: g[k] for k in ("y1", "y0", "mat", "angle", "q")}
        y1, _ = ctx.propagate_batch(st.trajs, **kw)
        return y1


def work(case):
    """Bytes: the mesh and every input and result once.  Operations: a ray's nearest hit as one box and one
    triangle test (about 70), its shading (about 50), for the primary rays and the third of them that bounce on."""
    kind = case["kind"]

    def mesh_bytes(name, facet):
        tris = 16 if name == "box_wing" else 40 if name == "box_wing_two_axis" else 125.0 / facet ** 2
        return tris * (6 * 3 * 4 / 2 + 16)

    def evals(n, N, bounces):
        return n * N * N * (1.0 + 0.35 * bounces) * 120.0

    if kind == "batch":
        sizes = [0.4, 0.2, 0.1, 0.05][: case["facets"]]
        flops = sum(evals(13 * 4, [256, 512, 333, 768][(k // 2) % 4], k % 3) for k in range(case["n"]))
        return {"bytes": sum(mesh_bytes("spacecraft", f) for f in sizes) + 96.0 * case["n"], "flops": flops}
    n, N, bounces = case.get("n", 1), case["N"], case["bounces"]
    size = mesh_bytes(case["mesh"], case.get("facet"))
    if kind == "arc":
        return {"bytes": size + 96.0 * n, "flops": evals(n * 13 * (3 + 2.5 * case["hours"]), N, bounces)}
    if kind == "adjoint":
        return {"bytes": size + 300.0, "flops": 4.0 * evals(4 * case["steps"], N, bounces)}
    if kind == "table_arcs":
        return {"bytes": 9600.0 + 96.0 * n, "flops": n * 13 * (3 + 2.5 * case["hours"]) * 600.0}
    if kind == "grad":
        return {"bytes": size + n * 300.0, "flops": 3.0 * evals(n, N, bounces)}
    bytes_ = size + n * 80.0 + (4.0 * n * N * N * (bounces + 1) if case.get("hits") else 0.0)
    return {"bytes": bytes_, "flops": evals(n, N, bounces) * (1.0 + 0.3 * case.get("diffuse", 0))}


# ------------------------------------------------------ the 64-bit evaluation
PAIRS = 1.2e11  # most (ray, triangle) pairs that exact() tries: about 20 s of 64-bit matrix products


def _pose(m, X, s, angles, mode):
    """Posed vertices: joint rotations composed down the tree (tracking: the panel normal towards s)."""
    dev = X.device
    eye = torch.eye(3, dtype=torch.float64, device=dev)
    t64 = lambda a: torch.tensor(np.asarray(a, np.float64), device=dev)  # noqa: E731
    M, T = [eye], [torch.zeros(3, dtype=torch.float64, device=dev)]
    for p in range(1, len(m.parent)):
        q, a = int(m.parent[p]), t64(m.axis[p])
        R = eye
        if float(a.abs().sum()) > 0.0:
            th = angles[p]
            if mode != "set":
                sl, n0 = M[q].T @ s, t64(m.normal0[p])
                n0 = n0 - (n0 @ a) * a
                th = torch.atan2(torch.linalg.cross(a, n0) @ sl, n0 @ sl) + (angles[p] if mode == "offset" else 0.0)
            th = torch.clamp(th, float(m.limits[p, 0]), float(m.limits[p, 1]))
            K = torch.zeros(3, 3, dtype=torch.float64, device=dev)
            K[0, 1], K[0, 2], K[1, 0], K[1, 2], K[2, 0], K[2, 1] = -a[2], a[1], a[2], -a[0], -a[1], a[0]
            R = eye + torch.sin(th) * K + (1.0 - torch.cos(th)) * (K @ K)
        pv = t64(m.pivot[p])
        M.append(M[q] @ R)
        T.append(M[q] @ (pv - R @ pv) + T[q])
    part = np.zeros(len(m.xyz), np.int64)
    part[m.tri.reshape(-1)] = np.repeat(m.tri_part, 3)
    part = torch.tensor(part, device=dev)
    return torch.einsum("vij,vj->vi", torch.stack(M)[part], X) + torch.stack(T)[part]


def _nearest(o, d, tri, skip, eps):
    """Nearest triangle of every ray beyond eps, -1 for none: side tests of the ray's line against the edges' lines
    as one matrix product, then the distance of those hit."""
    R, T = len(o), len(tri)
    best = torch.full((R,), math.inf, dtype=torch.float64, device=o.device)
    ids = torch.full((R,), T, dtype=torch.int64, device=o.device)
    a, b, c = tri[:, 0], tri[:, 1], tri[:, 2]
    edges = [torch.cat([torch.linalg.cross(p, q), q - p], dim=1).T.contiguous() for p, q in ((a, b), (b, c), (c, a))]
    nrm = torch.linalg.cross(b - a, c - a)
    line = torch.cat([d, torch.linalg.cross(o, d)], dim=1)
    step = max(1, int(1.5e8) // T)
    for r0 in range(0, R, step):
        e = [line[r0:r0 + step] @ w for w in edges]
        inside = ((e[0] >= 0) & (e[1] >= 0) & (e[2] >= 0)) | ((e[0] <= 0) & (e[1] <= 0) & (e[2] <= 0))
        ray, k = torch.nonzero(inside, as_tuple=True)
        ray = ray + r0
        t = ((a[k] - o[ray]) * nrm[k]).sum(1) / (d[ray] * nrm[k]).sum(1)
        ok = torch.isfinite(t) & (t > eps) & (k != skip[ray])
        ray, k, t = ray[ok], k[ok], t[ok]
        best.scatter_reduce_(0, ray, t, "amin")
        ties = t == best[ray]
        ids.scatter_reduce_(0, ray[ties], k[ties], "amin")
    return torch.where(ids == T, -1, ids)


def _stream(seed, c):
    """Uniforms in [0, 1) from outputs c of the SplitMix64 stream (int64 arithmetic wraps as the 64-bit words do)."""
    def i64(x):
        return x - (1 << 64) if x >= 1 << 63 else x

    def shr(z, k):
        return (z >> k) & ((1 << (64 - k)) - 1)

    z = seed + (c + 1) * i64(0x9E3779B97F4A7C15)
    z = (z ^ shr(z, 30)) * i64(0xBF58476D1CE4E5B9)
    z = (z ^ shr(z, 27)) * i64(0x94D049BB133111EB)
    return shr(z ^ shr(z, 31), 11).double() * 2.0 ** -53


def _basis(d):
    """The orthonormal basis (u, v) about d [..., 3]."""
    sg = torch.copysign(torch.ones_like(d[..., 2]), d[..., 2])
    a = -1.0 / (sg + d[..., 2])
    b = d[..., 0] * d[..., 1] * a
    u = torch.stack([1.0 + sg * d[..., 0] ** 2 * a, sg * b, -sg * d[..., 0]], dim=-1)
    return u, torch.stack([b, sg + d[..., 1] ** 2 * a, -d[..., 1]], dim=-1)


def _deposit(m, tri, ids, o, d, w, mat, side_mat):
    """Force, hit point, normal towards the ray, coefficients of rays (o, d) of weight w on the planes of triangles ids."""
    a, b, c = tri[ids, 0], tri[ids, 1], tri[ids, 2]
    n = torch.linalg.cross(b - a, c - a)
    n = n / n.norm(dim=1, keepdim=True)
    dn = (d * n).sum(1)
    front = dn < 0
    nf = torch.where(front[:, None], n, -n)
    rho = mat[torch.where(front, side_mat[ids, 0], side_mat[ids, 1])]
    t = ((a - o) * n).sum(1) / dn
    x = o + t[:, None] * d
    k = rho[:, 0] * dn.abs() + rho[:, 1] / 3.0
    f = w[:, None] * ((1.0 - rho[:, :1]) * d - 2.0 * k[:, None] * nf)
    return f, x, n, nf, dn, rho


def _evaluate(m, s, dist, N, bounces, mat, angles, mode, diffuse=0, seed=0):
    """Force, torque and hits [N*N, bounces+1] for one Sun direction; differentiable with the hits held."""
    dev = s.device
    s = s / s.norm()
    X = _pose(m, torch.tensor(np.asarray(m.xyz, np.float64), device=dev), s, angles, mode)
    tri = X[torch.tensor(m.tri, dtype=torch.int64, device=dev)]
    side_mat = torch.tensor(m.tri_mat, dtype=torch.int64, device=dev)
    cref = torch.tensor(np.asarray(m.c_ref, np.float64), device=dev)
    d0 = -s
    u, v = _basis(d0)
    pu, pv, pw = X @ u, X @ v, X @ d0
    umin, umax, vmin, vmax = pu[pu.argmin()], pu[pu.argmax()], pv[pv.argmin()], pv[pv.argmax()]
    wmin, wmax = pw.min().detach(), pw.max().detach()
    L = math.sqrt(float(((umax - umin) ** 2 + (vmax - vmin) ** 2 + (wmax - wmin) ** 2).detach()))
    pix = torch.arange(N, dtype=torch.float64, device=dev) + 0.5
    uc = (umin + pix * (umax - umin) / N).repeat_interleave(N)
    vc = (vmin + pix * (vmax - vmin) / N).repeat(N)
    o = uc[:, None] * u + vc[:, None] * v + (wmin - 1.0) * d0
    d, w = d0.expand(N * N, 3), torch.ones(N * N, dtype=torch.float64, device=dev)
    ray = torch.arange(N * N, device=dev)
    skip = torch.full((N * N,), -1, dtype=torch.int64, device=dev)
    hits = torch.full((N * N, bounces + 1), -1, dtype=torch.int32, device=dev)
    F, Tq = torch.zeros(3, dtype=torch.float64, device=dev), torch.zeros(3, dtype=torch.float64, device=dev)
    for seg in range(bounces + 1):
        with torch.no_grad():
            ids = _nearest(o, d, tri, skip, 0.0 if seg == 0 else 1e-9 * L)
        hits[ray, seg] = ids.int()
        on = ids >= 0
        ray, o, d, w, ids = ray[on], o[on], d[on], w[on], ids[on]
        f, x, n, nf, dn, rho = _deposit(m, tri, ids, o, d, w, mat, side_mat)
        F, Tq = F + f.sum(0), Tq + torch.linalg.cross(x - cref, f).sum(0)
        if seg == bounces:
            break
        if diffuse > 0:
            em = torch.nonzero(rho[:, 1] > 0.0).reshape(-1).repeat_interleave(diffuse)
            c = (ray[em] * (bounces + 1) + seg) * diffuse + torch.arange(len(em), device=dev) % diffuse
            u1, u2 = _stream(seed, 2 * c), _stream(seed, 2 * c + 1)
            t1, t2 = _basis(nf[em])
            ang = 2.0 * math.pi * u2
            dd = (u1.sqrt() * torch.cos(ang))[:, None] * t1 + (u1.sqrt() * torch.sin(ang))[:, None] * t2 \
                + (1.0 - u1).sqrt()[:, None] * nf[em]
            hit = _nearest(x[em], dd, tri, ids[em], 1e-9 * L)
            on = hit >= 0
            f, xd, *_ = _deposit(m, tri, hit[on], x[em][on], dd[on], (w * rho[:, 1])[em][on] / diffuse, mat, side_mat)
            F, Tq = F + f.sum(0), Tq + torch.linalg.cross(xd - cref, f).sum(0)
        w = w * rho[:, 0]
        on = w != 0.0
        ray, o, w, skip = ray[on], x[on], w[on], ids[on]
        d = (d - 2.0 * dn[:, None] * n)[on]
    scale = P0 / dist ** 2 * (umax - umin) * (vmax - vmin) / (N * N)
    return F * scale, Tq * scale, hits


def _rotation(q):
    w, x, y, z = q / q.norm()
    return torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y),
                        2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x),
                        2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)]).reshape(3, 3)


def exact(case, seed):
    # arcs: hundreds of evaluations each, far beyond the time there is
    if case["kind"] not in ("eval", "grad"):
        return None
    grad = case["kind"] == "grad"
    v = _arrays(dict(case, mode="offset") if grad else case, seed)
    m, N, bounces, n = v.mesh, case["N"], case["bounces"], case["n"]
    if n * N * N * float(m.n_tris) * (1.0 + 0.3 * bounces + 0.35 * case.get("diffuse", 0)) > PAIRS:
        return None
    dev = "cuda:0" if torch.cuda.is_available() else "cpu"
    leaf = [torch.tensor(a, dtype=torch.float64, device=dev, requires_grad=grad)
            for a in (v.quat, v.dirs, v.dist, m.mat, v.angles)]
    quat, dirs, dist, mat, angles = leaf
    acc, torque, hits = [], [], []
    for k in range(n):
        s, r = dirs[k], dist[k] if grad or case.get("dist") else 1.0
        if grad or case.get("quat"):
            R = _rotation(quat[k])
            s = R.T @ s
        F, T, h = _evaluate(m, s, r, N, bounces, mat, angles, v.mode, case.get("diffuse", 0), v.seed)
        if grad or case.get("quat"):
            F = R @ F / m.mass
        if grad:
            gF, gT = torch.tensor(v.g_acc[k], device=dev), torch.tensor(v.g_torque[k], device=dev)
            (gF @ F + gT @ T).backward()
        acc.append(F.detach()), torque.append(T.detach())
        hits.append(h)
    acc, torque = torch.stack(acc), torch.stack(torque)
    if grad:
        names = ("g_quat", "g_sun", "g_dist", "g_mat", "g_angles")
        return dict(zip(names, [x.grad for x in leaf]), acc=acc, torque=torque)
    out = dict(force=acc, torque=torque)
    if case.get("hits"):
        out["hits"] = torch.stack(hits)
    return out
