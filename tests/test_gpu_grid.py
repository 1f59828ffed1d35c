"""Segment queries through the uniform grids against the tree's: the megakernel walks
the grids of larger meshes, the wavefront form the tree, and both are to follow every
history alike."""
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


def test_megakernel_on_grids_matches_the_wavefront_on_trees():
    bvh = api.gadep_bvh_build(api.detmesh_build(W.COAX_P), 0)
    mats = api.Materials.default()
    n = 400_001
    a, b = (torch.empty(n, dtype=torch.float32, device="cuda") for _ in range(2))
    ra, sa = api.gadep_run(bvh, mats, W.COAX_POINT_25, 1332.0, n, edep_trace=a, opts=api.make_opts(variant=1))
    rb, sb = api.gadep_run(bvh, mats, W.COAX_POINT_25, 1332.0, n, edep_trace=b, opts=api.make_opts(variant=WAVEFRONT))
    assert torch.equal(a, b) and np.array_equal(sa, sb)
    assert [ra[k] for k in COUNTS] == [rb[k] for k in COUNTS]
