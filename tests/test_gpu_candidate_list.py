"""Pixels with more uncertain triangles than their own words hold share a list of their evaluation.  Where it
runs over, every one of them is traversed: the path of a pixel does not depend on the order of arrival."""
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


def sheaves(P, layers):
    """P x P small patches above a floor, each of mirrors through one axis that are a micrometre apart at their ends:
    all within the depth band of each other, and on one side the one whose box comes first lies last, so that a
    traversal's candidate list overflows.  On a grid of 4 P pixels a side a patch covers 4 x 4 pixel centres."""
    V = [(-1, -1, -0.5), (1, -1, -0.5), (1, 1, -0.5), (-1, 1, -0.5)]
    tri = [(0, 1, 2), (0, 2, 3)]
    a = 0.8 / P
    for i in range(P * P):
        x, y = (2 * (i // P) + 1) / P - 1, (2 * (i % P) + 1) / P - 1
        for k in range(layers):
            c, v = 1e-6 * (k + 1), len(V)
            V += [(x - a, y - a, -c), (x + a, y - a, c), (x + a, y + a, c), (x - a, y + a, -c)]
            tri += [(v, v + 1, v + 2), (v, v + 2, v + 3)]
    n = len(tri)
    return I.Mesh(np.array(V, float), np.array(tri, np.int32), np.zeros(n, np.int32), np.zeros((n, 2), np.int32),
                  np.array([[0.6, 0.2]]), **I._parts(1, [-1]), name="sheaves")


# three to six candidates a pixel (more on the diagonals of the patches, which traverse): a list that holds them,
# and one that runs over by far
@pytest.mark.parametrize("layers", [4, 5, 6, 7])
@pytest.mark.parametrize("P", [2, 16])
@pytest.mark.parametrize("n", [1, 5])
def test_paths_do_not_depend_on_arrival(ctx, layers, P, n):
    m, N = sheaves(P, layers), 4 * P
    mid = ctx.load_mesh(m)
    s = np.tile([[0.0, 0.0, 1.0]], (n, 1))
    Ft, Tt, Ht = ctx.eval_batch(mid, s, N=N, bounces=1, hits=True, traverse=True)
    traversed = ctx.eval_stats()["refined"]
    seen = set()
    for _ in range(6):
        F, T, H = ctx.eval_batch(mid, s, N=N, bounces=1, hits=True)
        refined = ctx.eval_stats()["refined"]
        seen.add((refined, F.tobytes(), T.tobytes()))
        assert np.array_equal(H, Ht)
        assert all(np.array_equal(F[0], F[k]) and np.array_equal(T[0], T[k]) for k in range(n))
    assert len(seen) == 1
    if P == 16:  # 28 entries a patch and more: ran over
        assert refined == traversed and (layers < 6 or refined > 1000 * n)
    else:
        assert refined <= n * P * P * 4 and (layers < 6 or refined < traversed)
    r = O.evaluate(m, s[0], N, 1)
    assert np.linalg.norm(F[0] - r["F"]) <= 1e-4 * np.linalg.norm(r["F"])
    ctx.free_mesh(mid)
