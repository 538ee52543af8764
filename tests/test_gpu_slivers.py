"""Triangles that are none in FP32 (their cross product, or its square, is zero) and are hit all the same:
the ray is traced again in FP64, in every trace path, and the force is the oracle's."""
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


def scene(kind):
    """A square mirror in the window, and above it a mirror sliver along a row of pixel centres (an odd grid's
    middle row, y = 0, or the row at y = 1 of a window from -2 to 2)."""
    y, h, x0, x1, half = {"underflow": (0.0, 1e-24, 0.1, 0.9, 1.0), "rounded": (1.0, 1e-12, 1.0, 1.8, 2.0)}[kind]
    V = np.array([(-half, -half, -1), (half, -half, -1), (half, half, -1), (-half, half, -1),
                  (x0, y, 0), (x1, y, 0), ((x0 + x1) / 2, y + h, 0)])
    tri = np.array([(0, 1, 2), (0, 2, 3), (4, 5, 6)], np.int32)
    return I.Mesh(V, tri, np.zeros(3, np.int32), np.zeros((3, 2), np.int32), np.array([[0.7, 0.2]]), **I._parts(1, [-1]),
                  name=kind)


@pytest.mark.parametrize("kind, N", [("underflow", 33), ("underflow", 65), ("rounded", 34)])
@pytest.mark.parametrize("n", [1, 3, 5])
@pytest.mark.parametrize("opts", ["plain", "traverse", "queue"])
def test_slivers_are_hit(ctx, kind, N, n, opts):
    from paper_2608_07307_gb300 import srp
    kw = {"plain": {}, "traverse": dict(traverse=True), "queue": dict(flags=srp.EVAL_QUEUE)}[opts]
    m = scene(kind)
    mid = ctx.load_mesh(m)
    s = np.tile([[0.0, 0.0, 1.0]], (n, 1))
    F, T, H = ctx.eval_batch(mid, s, N=N, bounces=2, hits=True, **kw)
    r = O.evaluate(m, s[0], N, 2, want_hits=True)
    assert (r["hits"][:, 0] == 2).sum() > 3  # the sliver
    assert ctx.eval_stats()["refined"] == n * (r["hits"][:, 0] == 2).sum()
    for k in range(n):
        h = np.asarray(H[k]).reshape(r["hits"].shape)
        # (the floor's diagonal runs through pixel centres: such a ray may go to either half)
        assert np.array_equal(h == 2, r["hits"] == 2) and np.array_equal(h >= 0, r["hits"] >= 0)
        assert np.linalg.norm(F[k] - r["F"]) <= 1e-4 * np.linalg.norm(r["F"])
        assert np.linalg.norm(T[k] - r["T"]) <= 1e-4 * np.linalg.norm(r["F"])
    ctx.free_mesh(mid)
