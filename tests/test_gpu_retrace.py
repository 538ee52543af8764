"""The FP64 re-trace of rays with more uncertain triangles than the candidate list
holds, by warps (few such rays) and by lanes (many), and the poses of deep and wide
kinematic trees, against the FP64 oracle."""
import math

import numpy as np
import pytest

from oracle import oracle as O
from paper_2608_07307_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_2608_07307_gb300 import srp
    c = srp.Context(0)
    yield c
    c.close()


def check_force(F, T, r, slack=0.0):
    fn = np.linalg.norm(r["F"])
    assert np.linalg.norm(F - r["F"]) <= 1e-4 * fn + slack, (F, r["F"])
    assert np.linalg.norm(T - r["T"]) <= 1e-4 * max(np.linalg.norm(r["T"]), fn) + slack * 1.5


def trough(a, copies):
    """A floor and, above it, a right-angled trough of side a whose two faces are
    `copies` coincident quads each: every ray into it has that many equal hits, twice."""
    V = [(-1, -1, -0.5), (1, -1, -0.5), (1, 1, -0.5), (-1, 1, -0.5),
         (-a, -a, a), (0, -a, 0), (0, a, 0), (-a, a, a), (a, -a, a), (a, a, a)]
    quads = [(0, 1, 2, 3)] + [(4, 5, 6, 7)] * copies + [(5, 8, 9, 6)] * copies
    tri = np.array([t for q in quads for t in ((q[0], q[1], q[2]), (q[0], q[2], q[3]))], np.int32)
    mats = np.array([[(k // 2) % 3] * 2 for k in range(len(tri))], np.int32)
    return I.Mesh(np.array(V, float), tri, np.zeros(len(tri), np.int32), mats,
                  np.array([[0.9, 0.1], [0.5, 0.3], [0.7, 0.2]]), **I._parts(1, [-1]), name="trough")


# one ray of a block and a few, as many as its warps take one by one and more, most of the grid
@pytest.mark.parametrize("a, N, bounces", [(0.02, 50, 2), (0.1, 61, 1), (0.25, 96, 2), (0.4, 128, 2), (0.9, 160, 1)])
def test_retraced_rays(ctx, a, N, bounces):
    m = trough(a, 20)
    mid = ctx.load_mesh(m)
    s = np.array([[0.03, 0.02, 1.0], [0.05, -0.04, 1.0]])
    s /= np.linalg.norm(s, axis=1, keepdims=True)
    F, T, H = ctx.eval_batch(mid, s, N=N, bounces=bounces, hits=True)
    assert ctx.eval_stats()["refined"] > 0
    for k in range(2):
        r = O.evaluate(m, s[k], N, bounces, want_hits=True, want_edge=True)
        diff = np.asarray(H[k]).reshape(r["hits"].shape) != r["hits"]
        bad = np.nonzero(diff.any(axis=1))[0]
        for ray in bad:
            assert r["edge"][ray, int(np.argmax(diff[ray]))] < 1e-6 * r["win"][6], (k, ray)
        # the floor's diagonal runs through pixel centres: such a ray may go to either triangle or, in
        # the oracle, between them; it moves the force by at most 2 P0 A_pix a segment, either way
        u0, u1, v0, v1 = r["win"][:4]
        check_force(F[k], T[k], r, len(bad) * 4 * (1 + bounces) * 4.56e-6 * (u1 - u0) * (v1 - v0) / N ** 2)
    F2, T2 = ctx.eval_batch(mid, s, N=N, bounces=bounces)
    assert np.array_equal(F, F2) and np.array_equal(T, T2)
    ctx.free_mesh(mid)


def tree(shape):
    """16 boxes: a chain of joints, a fan off the root, or pairs of arms on arms."""
    parts, joints = [], []
    for k in range(16):
        par = {"chain": k - 1, "fan": 0, "pairs": (k - 1) // 2}[shape] if k else -1
        x, y = (k % 4) * 1.1, (k // 4) * 1.1
        parts.append(I.box((x, y, 0.0), (x + 0.7, y + 0.5, 0.2), mat=((0.4, 0.2),)))
        ax = np.array([(1, 0, 0), (0, 1, 0), (0.6, 0, 0.8)][k % 3], float) * (0.0 if k in (0, 7) else 1.0)
        lim = (-math.pi, math.pi) if k % 2 else (-0.6, 0.9)
        joints.append(dict(parent=par, pivot=(x, y, 0.1), axis=tuple(ax), limits=lim, normal0=(0.0, 0.0, 1.0)))
    return I.merge(parts, joints)


@pytest.mark.parametrize("shape", ["chain", "fan", "pairs"])
@pytest.mark.parametrize("mode", ["track", "offset", "set"])
def test_poses_of_sixteen_parts(ctx, shape, mode):
    from paper_2608_07307_gb300 import srp
    m = tree(shape)
    mid = ctx.load_mesh(m)
    s = I.sun_dirs_uniform(3, seed=7)
    ang = 0.3 * np.sin(np.arange(16.0))
    kw, ok = {}, {}
    if mode != "track":
        ctx.set_panel_angles(mid, ang)
        kw = dict(panel_mode=srp.PANELS_SET if mode == "set" else srp.PANELS_TRACK_OFFSET)
        ok = dict(angles=ang) if mode == "set" else dict(offsets=ang)
    F, T = ctx.eval_batch(mid, s, N=64, bounces=1, **kw)
    for k in range(3):
        check_force(F[k], T[k], O.evaluate(m, s[k], 64, 1, **ok))
    ctx.free_mesh(mid)
