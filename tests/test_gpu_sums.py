"""Sums of energies against the histories themselves: a run that walks the grids adds its
deposits in FP64, a warp's 32 at a time in FP32.

Tolerance: the last of a warp's five FP32 additions is off by 0.29 of a unit in the last
place of its sum S (an even spread), less than 0.29 * 2^-23 S, and the additions before it
add up to as much again in half-sized sums: 5e-8 S per warp, independent from warp to warp.
Of 1e8 histories of the coax 1.2e7 deposit, in 4e5 warps or more: 8e-11 of the whole; five
times that is allowed to the rms of six runs."""
import math

import pytest

from paper_2605_25963_gb300 import api
from paper_2605_25963_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)


def test_active_deposits_on_grids_are_summed_as_accurately_as_warps_are():
    bvh = api.gadep_bvh_build(api.detmesh_build(W.COAX_P), 0)
    mats = api.Materials.default()
    n = 100_000_000
    trace = torch.empty(n, dtype=torch.float32, device="cuda")
    off = []
    for seed in range(6):
        r, _ = api.gadep_run(bvh, mats, W.COAX_POINT_25, 1332.0, n, edep_trace=trace, opts=api.make_opts(seed=11 + seed))
        want = trace.sum(dtype=torch.float64).item()
        off.append(r["sum_dep_active"] / want - 1.0)
    assert math.sqrt(sum(x * x for x in off) / len(off)) <= 4e-10, off
