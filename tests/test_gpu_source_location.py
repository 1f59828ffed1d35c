"""Point sources in every kind of place -- the world, inside solids, on a surface -- are
located alike by gadep_run and gadep_run_noalloc, which use the mesh's own index."""
import numpy as np
import pytest

from paper_2605_25963_gb300 import api, capi
from paper_2605_25963_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

COUNTS = ("n_hist", "n_fep", "n_zero", "n_over", "n_err", "n_segments", "n_interactions", "n_culled")


@pytest.mark.parametrize("n", [1, 5_003])
def test_sources_are_located_alike(n):
    mesh = api.detmesh_build(W.COAX_P)
    bvh = api.gadep_bvh_build(mesh, 0)
    mats = api.Materials.default()
    opts = api.make_opts()
    spec = torch.zeros(opts.n_bins, dtype=torch.int32, device="cuda")
    regions, refused = set(), 0
    for z in [25.0, 0.0] + [-0.37 - 3.1 * k for k in range(40)]:
        src = W.Source(kind=W.SRC_POINT, pos=(0.3, 0.2, z))
        try:
            regions.add(mesh.locate(src.pos))
        except capi.GadepError:
            refused += 1
            for call in (lambda: api.gadep_run(bvh, mats, src, 662.0, n, opts=opts),
                         lambda: api.gadep_run_noalloc(bvh, mats, src, 662.0, n, spec, opts=opts)):
                with pytest.raises(capi.GadepError, match="surface"):
                    call()
            continue
        r, s = api.gadep_run(bvh, mats, src, 662.0, n, opts=opts)
        q = api.gadep_run_noalloc(bvh, mats, src, 662.0, n, spec, opts=opts)
        q = q[0] if isinstance(q, tuple) else q
        assert [r[k] for k in COUNTS] == [q[k] for k in COUNTS] and r["n_hist"] == n
        assert np.array_equal(spec.cpu().numpy().view(np.uint32), s)
    assert -1 in regions and len(regions) >= 3 and refused >= 1
