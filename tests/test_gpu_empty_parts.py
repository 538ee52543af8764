"""Parts without triangles (a gimbal between two joints): no ray meets them, the tree check counts nothing in them."""
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


def craft(before, behind, moving):
    """A plate, and above it a box behind `before` links without triangles and in front of `behind` such links; with
    `moving` all of them turn.  Returns the mesh and its joint angles: the box's alone is not zero."""
    n, box = before + behind + 2, before + 1
    plate = I.box((-1, -1, -0.6), (1, 1, -0.5), h=0.25, mat=((0.6, 0.2),))
    b = I.box((-0.3, -0.3, -0.2), (0.3, 0.3, 0.2), h=0.2, mat=((0.6, 0.2),))
    V = np.concatenate([plate.xyz, b.xyz])
    tri = np.concatenate([plate.tri, b.tri + len(plate.xyz)]).astype(np.int32)
    part = np.array([0] * len(plate.tri) + [box] * len(b.tri), np.int32)
    ax, ang = np.zeros((n, 3)), np.zeros(n)
    if moving:
        ax[1:], ang[box] = (1.0, 0.0, 0.0), 0.3
    return I.Mesh(V, tri, part, np.zeros((len(tri), 2), np.int32), np.array([[0.6, 0.2]]),
                  **I._parts(n, [-1] + list(range(n - 1)), axis=ax), name="craft"), ang


DIRS = np.array([[1.0, 1.0, 1.0], [-1.0, 1.0, 1.0], [0.0, 0.0, 1.0], [0.3, -0.2, 0.9], [1.0, 0.0, 1.0]])


@pytest.mark.parametrize("before, behind", [(1, 0), (0, 1), (2, 2), (0, 14)])
@pytest.mark.parametrize("moving", [False, True])
def test_empty_links(ctx, before, behind, moving):
    """The same bits as without them: few evaluations and many, odd grids (rays through the body origin) too."""
    from paper_2608_07307_gb300 import srp
    out = []
    for m, ang in (craft(0, 0, moving), craft(before, behind, moving)):
        mid = ctx.load_mesh(m)
        ctx.set_panel_angles(mid, ang)
        rep = ctx.mesh_check(mid, np.array([0.1, 0.2, 1.0]))
        assert rep["leaf_refs"] == rep["n_tris"] == len(m.tri)
        assert rep["tris_not_once"] == rep["boxes_outside_parent"] == rep["tris_outside_leaf"] == rep["walk_bound"] == 0
        r = []
        for N in (31, 40):
            for kw in (dict(), dict(traverse=True), dict(n_diffuse=2)):
                for d in (DIRS, DIRS[:1], DIRS[3:]):
                    r += ctx.eval_batch(mid, d, N=N, bounces=2, hits=True, panel_mode=srp.PANELS_SET, **kw)
        out.append([np.array(x) for x in r])
        ctx.free_mesh(mid)
    assert all(np.array_equal(x, y) for x, y in zip(*out)) and np.abs(out[0][0]).sum() > 0
