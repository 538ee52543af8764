"""Primary segments of launches of few evaluations whose pixels all have uncertain triangles:
every lane of a tile writes a candidate column, and the warp settles all of them together."""
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


def sheet(N, on_vertices, z=0.0):
    """A mirror sheet over the window of N pixels a side: its vertices at the pixel centres
    (six triangles meet at each) or on the rows between them (two at each centre)."""
    c = -1.0 + (np.arange(N) + 0.5) * 2.0 / N
    x = np.concatenate([[-1.0], c, [1.0]])
    y = x if on_vertices else -1.0 + np.arange(N + 1) * 2.0 / N
    V = np.array([(a, b, z) for a in x for b in y])
    w = len(y)
    tri = []
    for i in range(len(x) - 1):
        for j in range(w - 1):
            p = i * w + j
            tri += [(p, p + w, p + w + 1), (p, p + w + 1, p + 1)]
    tri = np.array(tri, np.int32)
    return I.Mesh(V, tri, np.zeros(len(tri), np.int32), np.zeros((len(tri), 2), np.int32), np.array([[0.6, 0.2]]),
                  **I._parts(1, [-1]), name="sheet")


# two candidates a pixel; six, in the slot's list of further ones; more of those than the list holds
@pytest.mark.parametrize("N, on_vertices", [(8, False), (33, False), (64, False), (5, True), (11, True), (33, True)])
def test_every_pixel_uncertain(ctx, N, on_vertices):
    m = sheet(N, on_vertices)
    mid = ctx.load_mesh(m)
    s = np.tile([[0.0, 0.0, 1.0]], (8, 1))
    Fm, Tm, Hm = ctx.eval_batch(mid, s, N=N, bounces=1, hits=True)
    Ft, Tt, Ht = ctx.eval_batch(mid, s, N=N, bounces=1, hits=True, traverse=True)
    assert np.array_equal(Hm, Ht) and (np.asarray(Hm)[:, :, 0] >= 0).all()
    for n in (1, 2, 3):
        for _ in range(4):
            F, T, H = ctx.eval_batch(mid, s[:n], N=N, bounces=1, hits=True)
            assert np.array_equal(H, Hm[:n]) and np.array_equal(F, Fm[:n]) and np.array_equal(T, Tm[:n])
    r = O.evaluate(m, s[0], N, 1)
    assert np.linalg.norm(Fm[0] - r["F"]) <= 1e-4 * np.linalg.norm(r["F"])
    assert np.linalg.norm(Ft[0] - r["F"]) <= 1e-4 * np.linalg.norm(r["F"])
    ctx.free_mesh(mid)
