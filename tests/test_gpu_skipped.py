"""Evaluations skipped by a negative Sun distance, in contexts that have evaluated nothing yet: zero force
and torque in every trace path, and the other evaluations as without them."""
import numpy as np
import pytest

from paper_2608_07307_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mesh", ["box_wing", "spacecraft"])
@pytest.mark.parametrize("n", [1, 2, 7])
@pytest.mark.parametrize("opts", ["plain", "traverse", "queue", "diffuse", "diffuse_traverse"])
def test_skipped_in_a_new_context(mesh, n, opts):
    from paper_2608_07307_gb300 import srp
    m = I.box_wing() if mesh == "box_wing" else I.spacecraft(0.25)
    kw = dict(traverse="traverse" in opts, flags=srp.EVAL_QUEUE if opts == "queue" else 0,
              n_diffuse=2 if "diffuse" in opts else 0)
    s, d = I.sun_dirs_uniform(n, seed=5), np.ones(n)
    off = np.arange(n) % 3 == 0
    d[off] = -1.0
    with srp.Context(0) as c:
        mid = c.load_mesh(m)
        F, T = c.eval_batch(mid, s, sun_dist=d, N=40, bounces=1, **kw)
        assert (F[off] == 0).all() and (T[off] == 0).all()
        G, U = c.eval_batch(mid, s, sun_dist=np.ones(n), N=40, bounces=1, **kw)
        assert np.array_equal(F[~off], G[~off]) and np.array_equal(T[~off], U[~off]) and (np.abs(G).sum(axis=1) > 0).all()
