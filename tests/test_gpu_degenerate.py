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


# every trace path; launches of few evaluations and of many
@pytest.mark.parametrize("bad", list(BAD))
@pytest.mark.parametrize("n, k", [(1, 0), (3, 2), (6, 0)])
@pytest.mark.parametrize("opts", ["plain", "traverse", "queue", "diffuse"])
def test_no_direction_gives_nan(ctx, bad, n, k, opts):
    from paper_2608_07307_gb300 import srp
    m = I.box_wing()
    mid = ctx.load_mesh(m)
    kw = {"plain": {}, "traverse": dict(traverse=True), "queue": dict(flags=srp.EVAL_QUEUE), "diffuse": dict(n_diffuse=2)}[opts]
    s = I.sun_dirs_uniform(n, seed=5)
    a = ctx.eval_batch(mid, s, N=48, bounces=1, hits=True, **kw)
    s[k] = BAD[bad]
    F, T, H = ctx.eval_batch(mid, s, N=48, bounces=1, hits=True, **kw)
    st = ctx.eval_stats()
    assert np.isnan(F[k]).all() and np.isnan(T[k]).all() and (np.asarray(H)[k] == -1).all()
    assert st["evals"] == n and st["rays"] == n * 48 * 48
    for x, y in zip(a, (F, T, H)):
        assert all(np.array_equal(x[e], y[e]) for e in range(n) if e != k)
    ctx.free_mesh(mid)


@pytest.mark.parametrize("bad", ["nan", "one_nan"])
def test_gradient_of_a_direction_of_nans(ctx, bad):
    test_gradient_of_a_degenerate_direction(ctx, "box_wing", bad, 6, 0)
    test_gradient_of_a_degenerate_direction(ctx, "spacecraft", bad, 1, 0)


@pytest.mark.parametrize("scale", [1e-150, 1e-3, 1.7, 1e150])
def test_any_length(ctx, scale):
    mid = ctx.load_mesh(I.box_wing())
    s = I.sun_dirs_uniform(2, seed=5)
    F, T = ctx.eval_batch(mid, s, N=48, bounces=1)
    G, U = ctx.eval_batch(mid, s * scale, N=48, bounces=1)
    assert np.allclose(F, G, rtol=1e-9, atol=0) and np.isfinite(U).all()
    ctx.free_mesh(mid)


@pytest.mark.parametrize("bad", ["quaternion", "direction"])
def test_autograd_of_a_degenerate_attitude(ctx, bad):
    import torch
    from paper_2608_07307_gb300 import autograd as A
    m = I.box_wing()
    mid = ctx.load_mesh(m)

    def run(degenerate):
        t = lambda x: torch.tensor(np.asarray(x, np.float64), device="cuda", requires_grad=True)  # noqa: E731
        q, s = np.tile([0.9, 0.1, -0.3, 0.2], (5, 1)), I.sun_dirs_uniform(5, seed=9)
        if degenerate:
            (q if bad == "quaternion" else s)[2] = 0.0
        leaf = [t(q), t(s), t(np.ones(5)), t(m.mat), t(np.zeros(len(m.parent)))]
        acc, T = A.srp_accel_inertial(ctx, mid, *leaf, N=48, bounces=1)
        torch.autograd.backward([acc, T], [torch.ones_like(acc), torch.ones_like(T)])
        return [x.detach().cpu().numpy() for x in (acc, T, leaf[0].grad, leaf[1].grad)]

    a, b, c = run(False), run(True), run(False)
    for x, y, z in zip(a, b, c):
        assert np.isnan(y[2]).all()
        assert np.array_equal(x[[0, 1, 3, 4]], y[[0, 1, 3, 4]]) and np.array_equal(x, z)
    ctx.free_mesh(mid)
