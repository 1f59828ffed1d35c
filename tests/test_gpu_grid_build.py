"""Building the grids of meshes whose triangles are long or large and lie obliquely: their
boxes hold most of a grid's cells.  A build with a device copy may take twice the time of
the host's part (the trees) and 5 ms, the best of three each."""
import time

import numpy as np
import pytest

from paper_2605_25963_gb300 import api
from paper_2605_25963_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

from test_gpu_grid_ties import MEGA, box, on_grids_and_on_trees  # noqa: E402

A, B = np.cos(0.7), np.sin(0.7)
C, D = np.cos(0.9), np.sin(0.9)
TILT = np.array([[A, -B, 0], [B, A, 0], [0, 0, 1]]) @ np.array([[1, 0, 0], [0, C, -D], [0, D, C]])


def revolved(n, profile):
    """The solid that a profile of (radius, z) from the lower to the upper end encloses."""
    ang = 2.0 * np.pi * np.arange(n) / n
    xyz = [(0.0, 0.0, profile[0][1])] + [(r * np.cos(a), r * np.sin(a), z) for r, z in profile for a in ang] + \
          [(0.0, 0.0, profile[-1][1])]
    at = lambda j, i: 1 + j * n + i % n
    tri = []
    for i in range(n):
        tri += [(0, at(0, i + 1), at(0, i)), (len(xyz) - 1, at(len(profile) - 1, i), at(len(profile) - 1, i + 1))]
        for j in range(len(profile) - 1):
            tri += [(at(j, i), at(j, i + 1), at(j + 1, i + 1)), (at(j, i), at(j + 1, i + 1), at(j + 1, i))]
    return np.array(xyz), np.array(tri, np.int32)


def solids(parts, active, turn=TILT):
    xyz, tri, solid, base = [], [], [], 0
    for s, (x, t) in enumerate(parts):
        xyz.append(x @ turn.T)
        tri.append(t + base)
        solid.append(np.full(len(t), s, np.int32))
        base += len(x)
    n = len(parts)
    return api.detmesh_from_arrays(np.concatenate(xyz).astype(np.float32), np.concatenate(tri), np.concatenate(solid),
                                   [W.MAT_GE] * n, active, [-1] * n)


def best(f):
    out = []
    for _ in range(3):
        t = time.perf_counter()
        f()
        out.append(time.perf_counter() - t)
    return min(out)


@pytest.mark.parametrize("name", ["long", "large"])
def test_oblique_triangles_do_not_hold_up_the_build(name):
    if name == "long":
        mesh = solids([revolved(600, [(30.0, 0.0), (30.0, 60.0)])], [1])
    else:       # 200 boxes, each within the one before
        half = [30.0 - 0.1 * k for k in range(200)]
        mesh = solids([box((-h, -h, -h), (h, h, h), 1) for h in half], [1] * 200)
    api.gadep_bvh_build(mesh, 0)
    host, device = best(lambda: api.gadep_bvh_build(mesh, -1)), best(lambda: api.gadep_bvh_build(mesh, 0))
    assert device <= 2.0 * host + 5e-3, (host, device)


def test_oblique_mesh_on_grids_matches_the_trees():
    rings = [(7.0, 0.0), (14.0, 0.0), (22.0, 0.0)] + [(30.0, 60.0 * k / 8) for k in range(9)] + [(22.0, 60.0), (14.0, 60.0), (7.0, 60.0)]
    inner = [(0.9 * r, 1.0 + 0.95 * z) for r, z in rings]
    bvh = api.gadep_bvh_build(solids([revolved(150, rings), revolved(150, inner)], [0, 1]), 0)
    assert bvh.stats()["n_tri"] >= 8192
    src = W.Source(kind=W.SRC_POINT, pos=tuple(float(v) for v in TILT @ np.array([3.0, 2.0, 90.0])))
    grids, trees = on_grids_and_on_trees(bvh, src, 662.0, 500_000, variant=MEGA)
    assert grids[0] < 1.5 < trees[0]
    assert grids[1] == trees[1] and grids[1][4] == 0
    assert np.array_equal(grids[2], trees[2])


@pytest.mark.parametrize("rings,n,e_model,grids", [(True, 6_000_000, 0, True), (False, 6_000_000, 0, False),
                                                   (False, 60_000_000, 0, True), (True, 2_000_000, 1, True),
                                                   (False, 2_000_000, 1, False)])
def test_fans_walk_grids_in_large_runs_only(rings, n, e_model, grids):
    """A fan's centre is a long list in one cell, which holds up every iteration of a run."""
    inside = [(r, z) for r in (7.0, 14.0, 22.0) for z in (-60.0,)] if rings else []
    parts = []
    for k in range(5):
        wall = [(30.0 - k, -60.0 + k + (60.0 - 2 * k) * j / 4) for j in range(5)] if rings else [(30.0 - k, -60.0 + k), (30.0 - k, -k)]
        low, high = [(r - k, -60.0 + k) for r, _ in inside], [(r - k, -k) for r, _ in inside[::-1]]
        parts.append(revolved(100 if rings else 400, low + wall + high))
    bvh = api.gadep_bvh_build(solids(parts, [0, 0, 0, 0, 1], np.eye(3)), 0)
    assert 4096 <= bvh.stats()["n_tri"] <= 24576
    inst = api.make_instances([(662.0, W.Source(kind=W.SRC_POINT, pos=(1.0, 2.0, 8.0)), n, 0, [])])
    _, nodes, _, _, tested = api.gadep_count_work(bvh, api.Materials.default(), inst, api.make_opts(variant=2, e_model=e_model))
    assert (tested < 1.5 * nodes) == grids


def test_grids_report_their_memory():
    """Cells, lists and three permuted copies of the triangles: the copies are 144 B a triangle,
    and every region's grid has at least 4 B for each of 2^17 cells but for rounding up."""
    with_grids = api.gadep_bvh_build(api.detmesh_build(W.COAX_P), 0)
    n_tri, n_region = with_grids.stats()["n_tri"], with_grids.stats()["n_region"]
    free = torch.cuda.mem_get_info()[0]
    other = api.gadep_bvh_build(api.detmesh_build(W.COAX_P), 0)
    taken = free - torch.cuda.mem_get_info()[0]
    assert other.grid_bytes() == with_grids.grid_bytes() > 144 * n_tri + 2 * 131072 * n_region
    st = other.stats()
    # the mesh's blocks, each rounded up to 2 MB by the allocator
    assert other.grid_bytes() <= taken <= other.grid_bytes() + st["node_bytes"] + st["tri_bytes"] + 64 * n_tri + (20 << 20)
    assert api.gadep_bvh_build(api.detmesh_build(W.COAX_P), -1).grid_bytes() == 0
    assert api.gadep_bvh_build(api.detmesh_build(W.BARE_CYLINDER), 0).grid_bytes() == 0


def test_many_small_solids_share_the_smallest_grids():
    """2^22 cells for the smallest grids together, twice that with borders and rounding up, and
    160 cells a triangle for those of the world and of every triangle."""
    parts = []
    for k in range(150):
        xyz, tri = revolved(8, [(3.0, 0.0), (3.0, 6.0)])
        parts.append((xyz + 8.0 * np.array([k % 5, k // 5 % 5, k // 25]), tri))
    bvh = api.gadep_bvh_build(solids(parts, [1] * 150), 0)
    n_tri = bvh.stats()["n_tri"]
    assert n_tri >= 2048
    assert 0 < bvh.grid_bytes() <= 4 * (2 * (1 << 22) + 2 * 2 * 160 * n_tri) + 4 * 3 * 1000 * n_tri


@pytest.mark.parametrize("shape", ["boxes", "tilted boxes"])
def test_flat_meshes_have_no_grids(shape):
    """Boxes along the axes are the trees' best case."""
    parts = []
    for k in range(8):
        xyz, tri = box((0.0, 0.0, 0.0), (8.0, 8.0, 8.0), 6)
        xyz = np.round(xyz / (8.0 / 6)) * (8.0 / 6)             # without the dents
        parts.append((xyz + 10.0 * np.array([k & 1, k >> 1 & 1, k >> 2]), tri))
    bvh = api.gadep_bvh_build(solids(parts, [1] * 8, np.eye(3) if shape == "boxes" else TILT), 0)
    assert bvh.stats()["n_tri"] == 8 * 432
    assert (bvh.grid_bytes() > 0) == (shape == "tilted boxes")


@pytest.mark.parametrize("depth,n,e_model,grids", [(1, 6_000_000, 0, False), (3, 2_000_000, 1, False), (4, 2_000_000, 1, True),
                                                   (4, 6_000_000, 0, False), (4, 12_000_000, 0, True), (5, 6_000_000, 0, True)])
def test_wavefront_runs_walk_grids_in_deep_nests(depth, n, e_model, grids):
    """Half of the histories reach the can below the source."""
    parts = []
    for k in range(depth):
        r, top, low = 30.0 - k, -float(k), -60.0 + k
        rings = [0.25 * r, 0.5 * r, 0.75 * r]
        parts.append(revolved(300 if depth == 1 else 100, [(x, low) for x in rings] +
                              [(r, low + (top - low) * j / 4) for j in range(5)] + [(x, top) for x in rings[::-1]]))
    bvh = api.gadep_bvh_build(solids(parts, [0] * (depth - 1) + [1], np.eye(3)), 0)
    assert 4096 <= bvh.stats()["n_tri"] <= 24576 and bvh.grid_bytes() > 0
    inst = api.make_instances([(662.0, W.Source(kind=W.SRC_POINT, pos=(1.0, 2.0, 3.0)), n, 0, [])])
    _, nodes, _, _, tested = api.gadep_count_work(bvh, api.Materials.default(), inst, api.make_opts(variant=2, e_model=e_model))
    assert (tested < 1.5 * nodes) == grids
