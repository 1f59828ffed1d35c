"""Rays through an edge that two surfaces share meet both at one distance, and the order of
the tree's tests decides between them.  Runs on grids are to follow such histories as runs on
trees do.  A second instance far from the mesh, of one history, sends a plan to the trees: its
source lies beyond the distance that the grids' margins cover."""
import numpy as np
import pytest

from paper_2605_25963_gb300 import api, capi
from paper_2605_25963_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

MEGA, WAVEFRONT = 1, 2
COUNTS = ("n_hist", "n_fep", "n_zero", "n_over", "n_err", "n_segments", "n_interactions", "n_culled")
NEAR, FAR = (W.Source(kind=W.SRC_POINT, pos=(0.0, 0.0, z)) for z in (60.0, 3e6))


def box(lo, hi, n):
    """A closed box of n x n squares a face: (xyz, tri)."""
    at, xyz, tri = {}, [], []

    def vertex(p):
        if p not in at:
            at[p] = len(xyz)
            xyz.append([lo[a] + (hi[a] - lo[a]) * p[a] / n for a in range(3)])
        return at[p]

    for a in range(3):
        for side in (0, n):
            for i in range(n):
                for j in range(n):
                    q = []
                    for u, v in ((i, j), (i + 1, j), (i + 1, j + 1), (i, j + 1)):
                        p = [0, 0, 0]
                        p[a], p[(a + 1) % 3], p[(a + 2) % 3] = side, u, v
                        q.append(vertex(tuple(p)))
                    q = q if side else q[::-1]
                    tri += [(q[0], q[1], q[2]), (q[0], q[2], q[3])]
    return np.array(xyz, np.float32), np.array(tri, np.int32)


def boxes_on_an_edge(n, swap):
    """An active and a dead Ge box side by side, their common edge x = z = 0 under a thin Ge
    plate; swap: the dead one has the lower triangle ids.  The triangles are shuffled, so
    that the vertices sampled for the nesting lie off the common face."""
    left, right = box((-10.0, -7.0, -9.0), (0.0, 9.0, 0.0), n), box((0.0, -7.0, -9.0), (10.0, 9.0, 0.0), n)
    plate = box((-2.0, -2.0, 3.0), (2.0, 2.0, 3.0625), 6)
    parts, active = ([right, left, plate], [0, 1, 0]) if swap else ([left, right, plate], [1, 0, 0])
    for seed in range(50):
        rng = np.random.default_rng(seed)
        xyz, tri, solid, base = [], [], [], 0
        for s, (x, t) in enumerate(parts):
            xyz.append(x)
            tri.append(rng.permutation(t) + base)
            solid.append(np.full(len(t), s, np.int32))
            base += len(x)
        try:
            return api.detmesh_from_arrays(np.concatenate(xyz), np.concatenate(tri), np.concatenate(solid),
                                           [W.MAT_GE] * 3, active, [-1] * 3)
        except capi.GadepError:
            pass
    raise AssertionError("every order of the triangles samples a vertex of the common face")


def on_grids_and_on_trees(bvh, src, E, n, **kw):
    """The run beside a near and beside a far instance: (on grids, result, spectrum) each."""
    mats, out = api.Materials.default(), []
    for other in (NEAR, FAR):
        inst = api.make_instances([(E, src, n, 0, []), (E, other, 1, 1, [])])
        _, nodes, _, _, tested = api.gadep_count_work(bvh, mats, inst, api.make_opts(**kw))
        res, spec = api.gadep_run_batch(bvh, mats, inst, api.make_opts(**kw))
        # a tree's node has two boxes and more, a cell counts as one
        out.append((tested < 1.5 * nodes, [res[0][k] for k in COUNTS], spec[0].copy(), res[0]["sum_dep_active"]))
    return out


@pytest.mark.parametrize("swap", [0, 1])
def test_tracks_take_the_surface_that_the_tree_takes(swap):
    bvh = api.gadep_bvh_build(boxes_on_an_edge(10, swap), 0)
    src = W.Source(kind=W.SRC_PENCIL, pos=(0.0, 0.3, 20.0), dir=(0.0, 0.0, -1.0))
    grids, trees = on_grids_and_on_trees(bvh, src, 500.0, 2_000_000, variant=WAVEFRONT, e_model=1)
    assert grids[0] and not trees[0]
    assert grids[1] == trees[1]
    assert np.array_equal(grids[2], trees[2])
    assert grids[3] == pytest.approx(trees[3], rel=1e-7)      # FP32 block sums of the trees
