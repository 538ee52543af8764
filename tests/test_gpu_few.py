"""The trace of launches of few evaluations (a block per tile, a warp's rays walked
together) against the trace of launches of many (a lane per ray): the same hits,
force and torque bits, where the walk's lists and orders can go wrong."""
import numpy as np
import pytest

from paper_2608_07307_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_2608_07307_gb300 import srp
    c = srp.Context(0)
    yield c
    c.close()


def mirrors(mesh):
    """The mesh with coefficients that keep every ray going for all bounces."""
    return mesh.with_materials(np.tile([[0.9, 0.1]], (len(mesh.mat), 1)))


def crowd():
    """16 parts (the most there are): boxes of few and of many triangles side by side, some turning."""
    parts = [I.box((x, y, 0.0), (x + 0.8, y + 0.8, 0.5 + 0.1 * k), h=None if k % 3 else 0.1)
             for k, (x, y) in enumerate((i % 4, i // 4) for i in range(16))]
    joints = [dict(parent=-1)] + [dict(parent=0, pivot=(0, 0, 0), axis=(0, 0, 1) if k % 4 == 0 else (0, 0, 0))
                                  for k in range(1, 16)]
    return I.merge(parts, joints)


CASES = {
    # name: mesh, rays a side, bounces; the launch has few rays for its triangles (few_trace)
    "one_pixel": (lambda: mirrors(I.box_wing()), 1, 1),
    "ragged_tiles": (lambda: mirrors(I.box_wing()), 33, 4),
    "single_triangle_parts": (lambda: mirrors(I.merge([I.random_soup(1, k, scale=0.5) for k in range(5)])), 47, 2),
    "found_list_overflows": (lambda: mirrors(I.random_soup(900, 3, size=1.2)), 70, 2),
    "shared_edges": (lambda: mirrors(I.icosphere(4)), 65, 2),
    "sixteen_parts": (lambda: mirrors(crowd()), 90, 4),
    "mirror_trough": (lambda: I.v_trough(), 40, 4),
    "spacecraft": (lambda: mirrors(I.spacecraft(0.1)), 333, 2),
    "grazing_dish": (lambda: mirrors(I.spacecraft(0.05)), 512, 1),
}


@pytest.mark.parametrize("name", list(CASES))
def test_few_and_many_give_the_same_bits(ctx, name):
    make, N, bounces = CASES[name]
    mid = ctx.load_mesh(make())
    dirs = I.sun_dirs_uniform(6, seed=len(name))
    Fm, Tm, Hm = ctx.eval_batch(mid, dirs, N=N, bounces=bounces, hits=True)
    stm = ctx.eval_stats()
    hits = segments = 0
    for k in range(0, 6, 2 if N > 300 else 1):
        n = 1 + (k % 2 if N <= 300 else 0)
        F, T, H = ctx.eval_batch(mid, dirs[k:k + n], N=N, bounces=bounces, hits=True)
        m = len(F)
        assert np.array_equal(H, Hm[k:k + m]), (name, k)
        assert np.array_equal(F, Fm[k:k + m]) and np.array_equal(T, Tm[k:k + m]), (name, k)
        st = ctx.eval_stats()
        assert st["hits"][:bounces + 1] == [int((Hm[k:k + m, :, b] >= 0).sum()) for b in range(bounces + 1)], (name, k)
        hits += st["hits"][0]
    assert hits > 0 and stm["rays"] == 6 * N * N
    ctx.free_mesh(mid)


def test_walk_bound_reports_in_a_small_launch(ctx):
    from paper_2608_07307_gb300 import srp
    mid = ctx.load_mesh(mirrors(I.spacecraft(0.1)))
    d = I.sun_dirs_uniform(1, seed=4)
    F0, _ = ctx.eval_batch(mid, d, N=200, bounces=1)
    with pytest.raises(srp.SrpError) as e:
        ctx.eval_batch(mid, d, N=200, bounces=1, flags=srp.EVAL_TEST_WALK_BOUND)
    assert e.value.code == srp.SRP_ERR_STACK
    F1, _ = ctx.eval_batch(mid, d, N=200, bounces=1)
    assert np.array_equal(F0, F1)
    ctx.free_mesh(mid)
