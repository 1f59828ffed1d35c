"""Histories are handed to the megakernel's warps in chunks of what is left, or of a
stated size; whichever warp takes them, every history is the same."""
import numpy as np
import pytest

from paper_2605_25963_gb300 import api
from paper_2605_25963_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

MEGA = 1
COUNTS = ("n_hist", "n_fep", "n_zero", "n_over", "n_err", "n_segments", "n_interactions", "n_culled")


@pytest.mark.parametrize("n", [1, 31, 33, 4_097, 700_001])
@pytest.mark.parametrize("det,src", [("BARE_CYLINDER", W.BARE_POINT_100), ("DET2", W.COAX_POINT_25)])
def test_chunks_do_not_change_histories(det, src, n):
    bvh = api.gadep_bvh_build(api.detmesh_build(getattr(W, det)), 0)
    mats = api.Materials.default()
    out = []
    for chunk in (0, 1, 32, 300):
        trace = torch.full((n,), -7.0, dtype=torch.float32, device="cuda")
        r, s = api.gadep_run(bvh, mats, src, 662.0, n, edep_trace=trace, opts=api.make_opts(variant=MEGA, chunk=chunk))
        out.append(([r[k] for k in COUNTS], s, trace))
    for counts, s, trace in out[1:]:
        assert counts == out[0][0] and counts[0] == n
        assert np.array_equal(s, out[0][1]) and torch.equal(trace, out[0][2])


@pytest.mark.parametrize("det,src,e_model", [("BARE_CYLINDER", W.BARE_POINT_100, 0), ("DET2", W.TABLE4_SOURCE, 0),
                                             ("COAX_P", W.COAX_POINT_25, 1)])
def test_long_runs_are_the_sum_of_short_ones(det, src, e_model):
    """From 3 * 2^18 histories on, warps look for the histories that reach the scene together."""
    bvh = api.gadep_bvh_build(api.detmesh_build(getattr(W, det)), 0)
    mats = api.Materials.default()
    n, parts = (1 << 20) + 33, 2

    def run(m, at):
        trace = torch.full((m,), -7.0, dtype=torch.float32, device="cuda")
        r, s = api.gadep_run(bvh, mats, src, 1332.0, m, edep_trace=trace,
                             opts=api.make_opts(variant=MEGA, e_model=e_model, history_offset=at))
        return [r[k] for k in COUNTS], s.astype(np.int64), trace, r["sum_esc"] + r["sum_dep_all"]

    half = n // parts
    whole, a, b = run(n, 0), run(half, 0), run(n - half, half)
    assert whole[0] == [x + y for x, y in zip(a[0], b[0])]
    assert np.array_equal(whole[1], a[1] + b[1])
    assert torch.equal(whole[2], torch.cat([a[2], b[2]]))
    assert whole[3] == pytest.approx(n * 1332.0, rel=1e-6)
