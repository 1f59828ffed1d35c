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
    """A closed box of n x n squares a face: (xyz, tri).  The vertices within the faces at both
    ends of y and the lower end of z lie 0.02 inside by turns, for flat meshes have no grids."""
    at, xyz, tri = {}, [], []

    def vertex(p):
        if p not in at:
            at[p] = len(xyz)
            q = [lo[a] + (hi[a] - lo[a]) * p[a] / n for a in range(3)]
            for a, side, move in ((1, 0, 0.02), (1, n, -0.02), (2, 0, 0.02)):
                if p[a] == side and sum(p) % 2 and all(0 < p[b] < n for b in range(3) if b != a):
                    q[a] += move
            xyz.append(q)
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


def nested(parts, active):
    """Ge solids of the given surfaces.  The nesting is found from a few sampled vertices, which
    may not lie on another solid: the triangles are shuffled until they do not."""
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
                                           [W.MAT_GE] * len(parts), active, [-1] * len(parts))
        except capi.GadepError:
            pass
    raise AssertionError("every order of the triangles samples a vertex on another solid")


def box_in_a_box(swap):
    """A dead Ge box and an active one within it that shares the middle of its top face, within
    two shells."""
    outer, inner = box((-8.0, -8.0, -16.0), (8.0, 8.0, 0.0), 16), box((-4.0, -4.0, -8.0), (4.0, 4.0, 0.0), 8)
    shells = [box((-8.0 - d, -8.0 - d, -16.0 - d), (8.0 + d, 8.0 + d, d), 4) for d in (2.0, 1.0)]
    return nested(shells + [inner, outer], [0, 0, 1, 0]) if swap else nested(shells + [outer, inner], [0, 0, 0, 1])


def boxes_on_an_edge(n, swap):
    """An active and a dead Ge box side by side, their common edge x = z = 0 under a thin Ge
    plate; swap: the dead one has the lower triangle ids."""
    left, right = box((-10.0, -7.0, -9.0), (0.0, 9.0, 0.0), n), box((0.0, -7.0, -9.0), (10.0, 9.0, 0.0), n)
    plate = box((-2.0, -2.0, 3.0), (2.0, 2.0, 3.0625), 6)
    parts, active = ([right, left, plate], [0, 1, 0]) if swap else ([left, right, plate], [1, 0, 0])
    return nested(parts, active)


def on_grids_and_on_trees(bvh, src, E, n, **kw):
    """The run beside a near and beside a far instance: (boxes tested per node visited, counts,
    spectrum, active deposits) each.  A tree's node has two boxes and more, a cell counts as
    one of each; queries left to the tree count as the tree's."""
    mats, out = api.Materials.default(), []
    for other in (NEAR, FAR):
        inst = api.make_instances([(E, src, n, 0, []), (E, other, 1, 1, [])])
        _, nodes, _, _, tested = api.gadep_count_work(bvh, mats, inst, api.make_opts(**kw))
        res, spec = api.gadep_run_batch(bvh, mats, inst, api.make_opts(**kw))
        out.append((tested / nodes, [res[0][k] for k in COUNTS], spec[0].copy(), res[0]["sum_dep_active"]))
    return out


@pytest.mark.parametrize("swap", [0, 1])
def test_tracks_take_the_surface_that_the_tree_takes(swap):
    bvh = api.gadep_bvh_build(boxes_on_an_edge(18, swap), 0)
    src = W.Source(kind=W.SRC_PENCIL, pos=(0.0, 0.3, 20.0), dir=(0.0, 0.0, -1.0))
    grids, trees = on_grids_and_on_trees(bvh, src, 500.0, 2_000_000, variant=MEGA, e_model=1)
    assert grids[0] < trees[0]
    assert grids[1] == trees[1]
    assert np.array_equal(grids[2], trees[2])
    assert grids[3] == pytest.approx(trees[3], rel=1e-7)      # FP32 sums of a lane's histories


@pytest.mark.parametrize("pos,dir,grids", [((0.0, 0.0, 25.0), (0.0, 0.0, -1.0), False),        # the axis: vertices
                                           ((80.0, 0.0, -30.3), (-1.0, 0.0, 0.0), False),      # edges of the walls
                                           ((3.3, 1.7, 25.0), (0.0, 0.0, -1.0), True)])
@pytest.mark.parametrize("form", ["tracks", "gradients"])
def test_pencils_along_edges_take_the_trees(pos, dir, grids, form):
    """Every photon of such a pencil would leave every one of its queries to the tree."""
    bvh = api.gadep_bvh_build(api.detmesh_build(W.COAX_P), 0)
    mats = api.Materials.default()
    n = 300_000 if form == "tracks" else 4_300_000
    inst = api.make_instances([(662.0, W.Source(kind=W.SRC_PENCIL, pos=pos, dir=dir), n, 0, [])])
    if form == "tracks":
        _, nodes, _, _, tested = api.gadep_count_work(bvh, mats, inst, api.make_opts(variant=WAVEFRONT, e_model=1))
        assert (tested < 1.5 * nodes) == grids
        return
    plan = api.Plan(bvh, mats, inst, api.make_opts(variant=WAVEFRONT, n_group=4), grad=True)
    plan.launch()
    res = plan.results()[0][0]
    photons = sum(plan.queue_sizes())              # a photon is queued once per flight, or once per segment
    assert (photons < 0.6 * res["n_segments"]) == grids


@pytest.mark.parametrize("swap", [0, 1])
def test_surfaces_that_coincide_are_crossed_alike(swap):
    """A box within a box, with one face in common: every query through that face meets two
    surfaces of different solids at one distance."""
    bvh = api.gadep_bvh_build(box_in_a_box(swap), 0)
    src = W.Source(kind=W.SRC_DISK, pos=(0.3, 0.2, 12.0), radius=3.0)
    grids, trees = on_grids_and_on_trees(bvh, src, 662.0, 1_000_000, variant=WAVEFRONT, e_model=1)
    assert grids[0] < 1.5 < trees[0]
    assert grids[1] == trees[1] and grids[1][4] == 0
    assert np.array_equal(grids[2], trees[2])
