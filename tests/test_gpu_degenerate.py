"""Inputs that are not a direction or an attitude: they spoil their own evaluation and nothing else."""
import numpy as np
import pytest

from paper_2608_07307_gb300 import inputs as I

pytestmark = pytest.mark.gpu

NAN, INF = float("nan"), float("inf")
BAD = {"zero": [0, 0, 0], "nan": [NAN] * 3, "negative_nan": [-NAN] * 3, "one_nan": [0.3, NAN, 0.1], "inf": [INF, 0, -INF]}
MESHES = {"box_wing": I.box_wing, "spacecraft": lambda: I.spacecraft(0.25)}


@pytest.fixture(scope="module")
def ctx():
    from paper_2608_07307_gb300 import srp
    c = srp.Context(0)
    yield c
    c.close()


# launches of few evaluations and of many, the degenerate one alone, first and last
@pytest.mark.parametrize("mesh", list(MESHES))
@pytest.mark.parametrize("n, k", [(1, 0), (3, 2), (6, 0)])
@pytest.mark.parametrize("opts", ["plain", "traverse", "queue", "diffuse", "count"])
def test_rays_that_are_not_numbers_stay_in_the_tree(ctx, mesh, n, k, opts):
    """Every box lets a ray of NaNs in, unused child slots too: the walk ends by its bound, or finds
    nothing, and reads nothing outside the mesh."""
    from paper_2608_07307_gb300 import srp
    m = MESHES[mesh]()
    mid = ctx.load_mesh(m)
    kw = {"plain": {}, "traverse": dict(traverse=True), "queue": dict(flags=srp.EVAL_QUEUE), "diffuse": dict(n_diffuse=2),
          "count": dict(count=True)}[opts]
    s = I.sun_dirs_uniform(n, seed=5)
    a = ctx.eval_batch(mid, s, N=48, bounces=1, hits=True, **kw)
    for bad in BAD.values():
        t = s.copy()
        t[k] = bad
        try:
            F, T, H = ctx.eval_batch(mid, t, N=48, bounces=1, hits=True, **kw)
        except srp.SrpError as e:
            assert e.code == srp.SRP_ERR_STACK
        else:
            assert (np.asarray(H)[k] == -1).all()
            for x, y in zip(a, (F, T, H)):
                assert all(np.array_equal(x[e], y[e]) for e in range(n) if e != k)
    b = ctx.eval_batch(mid, s, N=48, bounces=1, hits=True, **kw)
    assert all(np.array_equal(x, y) for x, y in zip(a, b))
    ctx.free_mesh(mid)


# the window search of the gradient: no vertex has the bound of projections that are all NaN
@pytest.mark.parametrize("mesh", list(MESHES))
@pytest.mark.parametrize("bad", ["zero", "negative_nan", "inf"])
@pytest.mark.parametrize("n, k", [(1, 0), (3, 2), (6, 0)])
def test_gradient_of_a_degenerate_direction(ctx, mesh, bad, n, k):
    m = MESHES[mesh]()
    mid = ctx.load_mesh(m)
    rng = np.random.default_rng(n)
    s, gF, gT = I.sun_dirs_uniform(n, seed=5), rng.normal(size=(n, 3)), rng.normal(size=(n, 3))
    a = ctx.grad(mid, s, gF, gT, N=48, bounces=1)
    t = s.copy()
    t[k] = BAD[bad]
    b = ctx.grad(mid, t, gF, gT, N=48, bounces=1)
    keep = [e for e in range(n) if e != k]
    for name in ("F", "T", "sun"):
        assert np.isnan(b[name][k]).all(), (name, b[name][k])
        assert np.array_equal(a[name][keep], b[name][keep]), name
    assert np.isnan(b["mat"]).any()  # sums over the evaluations
    c = ctx.grad(mid, s, gF, gT, N=48, bounces=1)
    for name in a:
        assert np.array_equal(a[name], c[name]), name
    ctx.free_mesh(mid)
