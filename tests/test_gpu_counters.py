"""Traversal counters beyond 32 bits."""
import numpy as np
import pytest

from paper_2608_07307_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def deep_stack(n):
    """n triangles on top of each other over half of the window's uppermost 64th (the boxes cover all of it), and a
    small one in the opposite corner.  Their long edge keeps 1 / 128 pixel from the pixel centres of 8192 x 8192
    rays, so that none is uncertain; a ray beside them meets every box and no triangle."""
    z = np.linspace(0.0, 1e-4 * n, n)[:, None]
    corner = np.array([[-1.0, 1.0], [1.0, 1.0], [1.0, 1.0 - 1.0 / 32.0]])
    V = np.concatenate([np.tile(corner[None], (n, 1, 1)), np.tile(z[:, None], (1, 3, 1))], axis=2).reshape(-1, 3)
    V = np.concatenate([V, [(-1, -1, 0), (-0.99, -1, 0), (-1, -0.99, 0)]])
    tri = np.arange(3 * n + 3, dtype=np.int32).reshape(-1, 3)
    return I.Mesh(V, tri, np.zeros(n + 1, np.int32), np.zeros((n + 1, 2), np.int32), np.array([[0.3, 0.2]]),
                  **I._parts(1, [-1]), name="deep_stack")


def test_counts_beyond_32_bits():
    from paper_2608_07307_gb300 import srp
    with srp.Context(0) as c:
        mid = c.load_mesh(deep_stack(80000))
        c.eval_batch(mid, np.array([[0.0, 0.0, 1.0]]), N=8192, bounces=0, count=True, traverse=True)
        st = c.eval_stats()
    assert st["refined"] == 0
    # four boxes a node; half a million rays meet all of the stack's triangles, in nodes of at most four children
    assert st["box_tests"] == 4 * st["nodes_visited"]
    assert st["tris_tested"] > 80000 * (8192 * 128 // 2 - 8192)
    assert st["nodes_visited"] > st["tris_tested"] / 3.01
