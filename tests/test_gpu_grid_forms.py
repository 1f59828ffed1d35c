"""Which meshes walk grids, and the megakernel's runs where it matters: at the ends of the
range of sizes, on lists too long for the cell words, with gradients, and where its warps
look for histories that reach the scene together, with several instances and stated chunks."""
import numpy as np
import pytest

from paper_2605_25963_gb300 import api
from paper_2605_25963_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

from test_gpu_grid_build import revolved, solids  # noqa: E402
from test_gpu_grid_ties import COUNTS, FAR, MEGA, NEAR, box, nested, on_grids_and_on_trees  # noqa: E402

SOURCE = W.Source(kind=W.SRC_POINT, pos=(1.0, 2.0, 40.0))


@pytest.mark.parametrize("n,grids", [(26, False), (27, True), (82, True), (83, False)])
def test_the_megakernel_walks_grids_from_8192_to_81920_triangles(n, grids):
    """A box of n x n squares a face: 8,112, 8,748, 80,688 and 82,668 triangles."""
    bvh = api.gadep_bvh_build(nested([box((-20.0, -21.0, -30.0), (22.0, 20.0, 0.0), n)], [1]), 0)
    assert bvh.stats()["n_tri"] == 12 * n * n
    near, far = on_grids_and_on_trees(bvh, SOURCE, 662.0, 100_000, variant=MEGA)
    assert (near[0] < 1.5) == grids and far[0] > 1.5
    assert near[1] == far[1] and near[1][4] == 0
    assert np.array_equal(near[2], far[2])


@pytest.mark.parametrize("n,grids", [(13, False), (14, True)])
def test_grids_are_built_from_2048_triangles(n, grids):
    bvh = api.gadep_bvh_build(nested([box((-20.0, -21.0, -30.0), (22.0, 20.0, 0.0), n)], [1]), 0)
    assert (bvh.grid_bytes() > 0) == grids


@pytest.mark.parametrize("e_model", [0, 1])
def test_long_lists(e_model):
    """Cans with fans of 1,100 triangles as end faces, whose centres are one cell each, the
    source above them; the length of such a list is its first entry."""
    cans = [revolved(1100, [(30.0 - k, -60.0 + k), (30.0 - k, -k)]) for k in range(2)]
    bvh = api.gadep_bvh_build(solids(cans, [0, 1], np.eye(3)), 0)
    assert bvh.stats()["n_tri"] >= 8192
    src = W.Source(kind=W.SRC_DISK, pos=(0.0, 0.0, 5.0), radius=0.5)
    grids, trees = on_grids_and_on_trees(bvh, src, 662.0, 200_000, variant=MEGA, e_model=e_model)
    assert grids[0] < 1.5 < trees[0]
    assert grids[1] == trees[1] and grids[1][4] == 0
    assert np.array_equal(grids[2], trees[2])


def test_a_long_thin_rod():
    """Thousands of cells along one axis, two dozen across."""
    rod = revolved(64, [(0.25, -70.0)] + [(0.5, -70.0 + 120.0 * k / 70) for k in range(71)] + [(0.25, 50.0)])
    bvh = api.gadep_bvh_build(solids([rod], [1], np.eye(3)), 0)
    assert bvh.stats()["n_tri"] >= 8192
    src = W.Source(kind=W.SRC_DISK, pos=(0.1, 0.2, 51.0), radius=0.6)
    grids, trees = on_grids_and_on_trees(bvh, src, 122.0, 500_000, variant=MEGA)
    assert grids[0] < 1.5 < trees[0]
    assert grids[1] == trees[1] and grids[1][4] == 0
    assert np.array_equal(grids[2], trees[2])


def test_megakernel_gradients_on_grids_match_the_trees():
    bvh = api.gadep_bvh_build(api.detmesh_build(W.GRAD_DET), 0)
    mats, out = api.Materials.default(), []
    opts = api.make_opts(variant=MEGA, n_group=4)
    for other in (NEAR, FAR):
        inst = api.make_instances([(1332.0, W.GRAD_SOURCE, 200_000, 0, [1.1, 0.9, 1.0, 0.8]), (662.0, other, 1, 1, [])])
        _, nodes, _, _, tested = api.gadep_count_work(bvh, mats, inst, opts)
        res, spec, d, ds = api.gadep_grad(bvh, mats, inst, opts)
        out.append((tested / nodes, [res[0][k] for k in COUNTS], spec[0].copy(), d[0], ds[0]))
    grids, trees = out
    assert grids[0] < 1.5 < trees[0]
    assert grids[1] == trees[1] and np.array_equal(grids[2], trees[2])
    # FP64 sums of the same scores in another order
    assert np.allclose(grids[3], trees[3], rtol=1e-9) and np.allclose(grids[4], trees[4], rtol=1e-9)


@pytest.mark.parametrize("chunk", [0, 1, 1000, 300_000])
def test_common_births_of_several_instances(chunk):
    """Together 2^20 histories or so, in counts that are no multiples of a warp, one of none;
    each by itself is too short a run for common births."""
    bvh = api.gadep_bvh_build(api.detmesh_build(W.DET2), 0)
    mats = api.Materials.default()
    srcs = [W.TABLE4_SOURCE, W.COAX_POINT_25, W.Source(kind=W.SRC_DISK, pos=(5.0, 0.0, 60.0), radius=20.0), W.TABLE4_SOURCE,
            W.Source(kind=W.SRC_PENCIL, pos=(3.0, 4.0, 80.0), dir=(0.0, 0.0, -1.0))]
    counts = [400_003, 0, 250_031, 1, 400_017]
    items = [(300.0 + 200.0 * i, s, n, i, []) for i, (s, n) in enumerate(zip(srcs, counts))]
    opts = api.make_opts(variant=MEGA, chunk=chunk)
    res, spec = api.gadep_run_batch(bvh, mats, api.make_instances(items), opts)
    for i, (E, s, n, _, _) in enumerate(items):
        r, want = api.gadep_run(bvh, mats, s, E, n, instance=i, opts=api.make_opts(variant=MEGA))
        assert [res[i][k] for k in COUNTS] == [r[k] for k in COUNTS]
        assert np.array_equal(spec[i], want)
        assert res[i]["sum_dep_all"] + res[i]["sum_esc"] == pytest.approx(n * E, rel=1e-6)
