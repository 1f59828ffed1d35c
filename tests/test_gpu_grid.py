"""Segment queries through the uniform grids against the tree's: a run of many
histories walks the grids in the trace kernel, runs of fewer histories of the same
id range take the tree, and both are to follow every history alike, so that the
tallies and spectra of the parts add up to those of the whole, exactly.  The meshes
lie at both ends of the range that the rule on sizes gives the grids."""
import dataclasses

import numpy as np
import pytest

from paper_2605_25963_gb300 import api
from paper_2605_25963_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

WAVEFRONT = 2
COUNTS = ("n_hist", "n_fep", "n_zero", "n_over", "n_err", "n_segments", "n_interactions", "n_culled")


@pytest.mark.parametrize("n_theta,E", [(40, 59.5), (128, 1332.0), (144, 662.0)])
def test_grid_run_is_the_sum_of_tree_runs(n_theta, E):
    bvh = api.gadep_bvh_build(api.detmesh_build(dataclasses.replace(W.COAX_P, n_theta=n_theta)), 0)
    assert 4096 <= bvh.stats()["n_tri"] <= 24576
    mats = api.Materials.default()
    n, parts = 4_800_003, 6                       # a quarter reach the scene: 1.2e6, and 2e5 a part
    r, spec = api.gadep_run(bvh, mats, W.COAX_POINT_25, E, n, opts=api.make_opts(variant=WAVEFRONT))
    at, got, total = 0, np.zeros_like(spec), dict.fromkeys(COUNTS, 0)
    for i in range(parts):
        m = n // parts if i < parts - 1 else n - at
        q, s = api.gadep_run(bvh, mats, W.COAX_POINT_25, E, m, opts=api.make_opts(variant=WAVEFRONT, history_offset=at))
        got += s
        for k in COUNTS:
            total[k] += q[k]
        at += m
    assert {k: r[k] for k in COUNTS} == total
    assert np.array_equal(spec, got)
    assert r["n_err"] == 0 and r["sum_dep_all"] + r["sum_esc"] == pytest.approx(n * E, rel=1e-6)


def test_grid_gradients_match_the_tree():
    """Scores accumulated by the trace kernel along a flight (grids: 4.4e6 histories in
    one call) and by physics segment by segment (1.1e6 a call)."""
    bvh = api.gadep_bvh_build(api.detmesh_build(W.GRAD_DET), 0)
    mats = api.Materials.default()
    scales = [1.1, 0.9, 1.0, 0.8]
    items = [(E, W.GRAD_SOURCE, 1_100_000, i, scales) for i, E in enumerate(W.GRAD_ENERGIES)]
    opts = api.make_opts(n_group=4, variant=WAVEFRONT)
    res, spec, d, ds = api.gadep_grad(bvh, mats, api.make_instances(items), opts)
    for i, it in enumerate(items):
        r1, s1, d1, ds1 = api.gadep_grad(bvh, mats, api.make_instances([it]), opts)
        assert [res[i][k] for k in COUNTS] == [r1[0][k] for k in COUNTS]
        assert np.array_equal(spec[i], s1[0])
        assert np.allclose(d[i], d1[0], rtol=1e-9) and np.allclose(ds[i], ds1[0], rtol=1e-9)


@pytest.mark.parametrize("n_theta,e_model", [(60, 1), (128, 0)])
def test_megakernel_on_grids_matches_the_wavefront_on_trees(n_theta, e_model):
    """6480 triangles: the wavefront form of electron runs walks grids, the megakernel the
    tree; 20,088: the megakernel walks grids, this wavefront run the tree."""
    bvh = api.gadep_bvh_build(api.detmesh_build(dataclasses.replace(W.COAX_P, n_theta=n_theta)), 0)
    mats = api.Materials.default()
    n = 400_001
    a, b = (torch.empty(n, dtype=torch.float32, device="cuda") for _ in range(2))
    ra, sa = api.gadep_run(bvh, mats, W.COAX_POINT_25, 1332.0, n, edep_trace=a, opts=api.make_opts(variant=1, e_model=e_model))
    rb, sb = api.gadep_run(bvh, mats, W.COAX_POINT_25, 1332.0, n, edep_trace=b, opts=api.make_opts(variant=WAVEFRONT, e_model=e_model))
    assert torch.equal(a, b) and np.array_equal(sa, sb)
    assert [ra[k] for k in COUNTS] == [rb[k] for k in COUNTS]
