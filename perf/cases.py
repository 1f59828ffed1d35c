"""The work that users of the framework have it do, as cases that can be timed.

A case is a plain dict.  "kind" names the public entry point it goes through:

    hits      gadep_nearest_hit on a user's own mesh (detmesh_from_arrays)
    run       gadep_run, host spectrum
    noalloc   gadep_run_noalloc, device spectrum
    batch     gadep_run_batch, one call over many instances
    grad      gadep_grad, density-perturbation gradients
    plan      Plan.launch + Plan.results, the form that is launched repeatedly

"det" names the detector of paper_2605_25963_gb300.workloads (its sizes and its
source positions are used as they are there; "n_theta" changes the segments per
circle, as the mesh-density sweep of the benchmark does).  "n" is the number of
histories (rays for hits) per instance, "energy" in keV.
"""
import dataclasses
import math

import numpy as np
import torch

from paper_2605_25963_gb300 import api
from paper_2605_25963_gb300 import workloads as W

# detector, source, and the segments (surface queries) an emitted history takes on
# average: most histories of a distant point source end at birth
SETUPS = {
    "bare": (W.BARE_CYLINDER, W.BARE_POINT_100, 1.1),
    "coax": (W.COAX_P, W.COAX_POINT_25, 2.2),
    "coax_n": (W.COAX_N, W.COAX_POINT_25, 2.2),
    "det2": (W.DET2, W.TABLE4_SOURCE, 1.05),
    "prism": (W.GRAD_DET, W.GRAD_SOURCE, 3.7),
}


def listed():
    return [
        # A handful of geometry queries (is this point inside, what does this ray meet
        # first): the smallest call there is, bound by its latency.
        dict(name="hits_2e3", kind="hits", n=2_000, n_theta=48, regions=False),
        # Ray casting through a detector in bulk (attenuation maps, path lengths), with
        # the region of every origin known.
        dict(name="hits_1e6_regions", kind="hits", n=1_000_003, n_theta=128, regions=True),
        # A quick look at a bare crystal: the smallest transport call, mostly fixed cost.
        dict(name="run_bare_2e4", kind="run", det="bare", energy=662.0, n=20_000),
        # The bare-cylinder workload as the configuration has it: 1e6 histories, 662 keV.
        dict(name="run_bare_1e6", kind="run", det="bare", energy=662.0, n=1_000_000),
        # One energy of the paper's Table 4 experiment (source at 250 mm, 1e7 particles).
        dict(name="run_det2_250mm_1e7", kind="run", det="det2", energy=778.9, n=10_000_000),
        # A run inside an application that owns the device memory; a low line, an odd count.
        dict(name="noalloc_coax_300003", kind="noalloc", det="coax", energy=122.0, n=300_003),
        # An ordinary efficiency point on the coaxial detector.
        dict(name="run_coax_1e7_662", kind="run", det="coax", energy=662.0, n=10_000_000),
        # The headline's share for one energy: 1e8 histories on the coaxial detector.
        dict(name="run_coax_1e8_1332", kind="run", det="coax", energy=1332.0, n=100_000_000),
        # Charged-particle tracks on.
        dict(name="electrons_coax_5e6", kind="run", det="coax", energy=1332.0, n=5_000_000, e_model=1),
        # The batched calibration matrix, 40 energies x 3 sources with uneven counts, at a
        # tenth of the workload's histories.
        dict(name="batch_120", kind="batch", det="batch", lo=1e5, hi=5e6),
        # Gradients with respect to the four density groups, volume source.
        dict(name="grad_prism_4x3e6", kind="grad", det="prism", n=3_000_000),
        # A fine mesh (512 segments, 216,684 triangles) under a volume source, a plan that
        # is launched again and again; eight energies.
        dict(name="plan_prism_512_8x2e6", kind="plan", det="prism", n_theta=512, n_phi=20, n=2_000_000, n_energy=8),
    ]


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["hits", "run", "run", "run", "run", "noalloc", "batch", "grad", "plan"])
    if kind == "hits":
        return dict(kind=kind, n=int(_log_uniform(rng, 2e3, 1e6)), n_theta=rng.randint(24, 128),
                    regions=rng.random() < 0.5)
    if kind == "run":
        det = rng.choice(["bare", "coax", "coax", "coax_n", "det2", "prism"])
        hi = {"bare": 1e8, "coax": 1e8, "coax_n": 1e8, "det2": 1e8, "prism": 1.5e7}[det]
        c = dict(kind=kind, det=det, energy=round(_log_uniform(rng, 59.5, 1836.0), 2),
                 n=int(_log_uniform(rng, 2e4, hi)))
        if det not in ("bare", "det2"):
            if rng.random() < 0.25:
                c["e_model"] = 1
                c["n"] = min(c["n"], 5_000_000)
            c["n_theta"] = rng.randint(32, 256)
        return c
    if kind == "noalloc":
        return dict(kind=kind, det=rng.choice(["bare", "coax", "det2"]), energy=round(_log_uniform(rng, 59.5, 1836.0), 2),
                    n=int(_log_uniform(rng, 2e4, 2e6)))
    if kind == "batch":
        hi = _log_uniform(rng, 1e5, 5e6)
        return dict(kind=kind, det="batch", lo=hi / 50.0, hi=hi)
    if kind == "grad":
        return dict(kind=kind, det="prism", n=int(_log_uniform(rng, 2e5, 3e6)), n_theta=rng.randint(32, 160))
    return dict(kind=kind, det=rng.choice(["coax", "prism"]), n_theta=rng.randint(64, 384), n_phi=rng.randint(10, 20),
                n=int(_log_uniform(rng, 1e5, 2e6)), n_energy=rng.randint(1, 8))


# ---------------------------------------------------------------- a user's own mesh

# nested cylinders of revolution: (radius, z low, z high, material, active): an Al can,
# its vacuum, a dead Ge layer and the active Ge
CYLINDERS = ((38.0, -120.0, 0.0, W.MAT_AL, 0), (37.0, -119.0, -1.0, W.MAT_VACUUM, 0),
             (30.5, -68.0, -6.0, W.MAT_GE, 0), (29.8, -67.3, -6.7, W.MAT_GE, 1))


def _revolved_mesh(n_theta):
    """(xyz, tri, solid) of the nested cylinders: end faces of three rings and a small
    fan, side walls of four bands."""
    ang = 2.0 * np.pi * np.arange(n_theta) / n_theta
    xyz, tri, solid = [], [], []
    for s, (R, z0, z1, _, _) in enumerate(CYLINDERS):
        prof = [(R * f, z0) for f in (0.25, 0.5, 0.75)] + [(R, z0 + (z1 - z0) * k / 4.0) for k in range(5)] + \
               [(R * f, z1) for f in (0.75, 0.5, 0.25)]
        base = len(xyz)
        xyz.append((0.0, 0.0, z0))
        for r, z in prof:
            xyz += [(r * math.cos(a), r * math.sin(a), z) for a in ang]
        xyz.append((0.0, 0.0, z1))
        top = len(xyz) - 1
        ring = lambda j, i: base + 1 + j * n_theta + i % n_theta
        m = len(prof)
        for i in range(n_theta):
            tri.append((base, ring(0, i + 1), ring(0, i)))
            tri.append((top, ring(m - 1, i), ring(m - 1, i + 1)))
            for j in range(m - 1):
                a, b, c, d = ring(j, i), ring(j, i + 1), ring(j + 1, i), ring(j + 1, i + 1)
                tri += [(a, b, d), (a, d, c)]
        solid += [s] * (len(tri) - len(solid))
    return np.array(xyz, np.float32), np.array(tri, np.int32), np.array(solid, np.int32)


def _rays(case, seed):
    """Rays as a user casts them: from the source side towards the detector, and from
    the active crystal outwards; their regions (0 world, s + 1 solid s)."""
    rng = np.random.default_rng(seed)
    n = case["n"]
    rays = np.zeros((n, 8), np.float32)
    inside = rng.random(n) < 0.5
    phi, r = rng.uniform(0, 2 * np.pi, n), np.sqrt(rng.random(n))
    o = np.column_stack([r * 35.0 * np.cos(phi), r * 35.0 * np.sin(phi), rng.uniform(5.0, 45.0, n)])
    o[inside] = np.column_stack([r * 28.0 * np.cos(phi), r * 28.0 * np.sin(phi), rng.uniform(-65.0, -9.0, n)])[inside]
    d = rng.normal(size=(n, 3))
    d[~inside, 2] = -np.abs(d[~inside, 2])
    d /= np.linalg.norm(d, axis=1, keepdims=True)
    rays[:, 0:3], rays[:, 4:7] = o, d
    rays[:, 7] = np.full(n, -1, np.int32).view(np.float32)
    return rays, np.where(inside, 4, 0).astype(np.int32)


# ---------------------------------------------------------------- prepare, run

def _detector(case):
    if case["det"] == "batch":
        return W.BATCH_DET
    det = SETUPS[case["det"]][0]
    new = {k: case[k] for k in ("n_theta", "n_phi") if k in case}
    return dataclasses.replace(det, **new) if new else det


def _instances(case):
    if case["kind"] == "batch":
        items = W.batch_instances(lo=case["lo"], hi=case["hi"])
        return [(E, W.BATCH_SOURCES[s], n, i, [1.0, 1.0, 1.0, sc]) for i, (E, s, n, sc) in enumerate(items)]
    src = SETUPS[case["det"]][1]
    energies = W.GRAD_ENERGIES if case["kind"] == "grad" else W.STRESS_ENERGIES[:case["n_energy"]]
    return [(E, src, case["n"], i, []) for i, E in enumerate(energies)]


def prepare(case, seed):
    kind = case["kind"]
    st = dict(kind=kind, mats=None)
    if kind == "hits":
        xyz, tri, solid = _revolved_mesh(case["n_theta"])
        mesh = api.detmesh_from_arrays(xyz, tri, solid, [c[3] for c in CYLINDERS], [c[4] for c in CYLINDERS],
                                       [-1] * len(CYLINDERS))
        rays, reg = _rays(case, seed)
        st["rays"] = torch.from_numpy(rays).cuda()
        st["regions"] = torch.from_numpy(reg).cuda() if case["regions"] else None
        st["bvh"] = api.gadep_bvh_build(mesh, 0)
        return st
    st["bvh"] = api.gadep_bvh_build(api.detmesh_build(_detector(case)), 0)
    st["mats"] = api.Materials.default()
    kw = dict(seed=1 + seed, e_model=case.get("e_model", 0))
    if kind == "grad":
        kw["n_group"] = W.GRAD_N_GROUP
    st["opts"] = api.make_opts(**kw)
    if kind in ("run", "noalloc"):
        st["src"], st["energy"], st["n"] = SETUPS[case["det"]][1], case["energy"], case["n"]
        if kind == "noalloc":
            st["spectrum"] = torch.zeros(st["opts"].n_bins, dtype=torch.int32, device="cuda")
    else:
        st["instances"] = api.make_instances(_instances(case))
        if kind == "plan":
            st["plan"] = api.Plan(st["bvh"], st["mats"], st["instances"], st["opts"])
    return st


def _columns(results):
    """The result records of many instances, one array per field."""
    return {k: np.array([r[k] for r in results]) for k in results[0]}


def run(st):
    kind = st["kind"]
    if kind == "hits":
        return api.gadep_nearest_hit(st["bvh"], st["rays"], regions=st["regions"])
    if kind == "run":
        return api.gadep_run(st["bvh"], st["mats"], st["src"], st["energy"], st["n"], opts=st["opts"])
    if kind == "noalloc":
        r = api.gadep_run_noalloc(st["bvh"], st["mats"], st["src"], st["energy"], st["n"], st["spectrum"],
                                  opts=st["opts"])
        return r, st["spectrum"]
    if kind == "batch":
        res, spec = api.gadep_run_batch(st["bvh"], st["mats"], st["instances"], st["opts"])
        return _columns(res), spec
    if kind == "grad":
        res, spec, d, ds = api.gadep_grad(st["bvh"], st["mats"], st["instances"], st["opts"])
        return _columns(res), spec, d, ds
    st["plan"].launch()
    res, spec, _, _ = st["plan"].results()
    return _columns(res), spec


# ---------------------------------------------------------------- work, exact

# Operations one segment cannot do without: one ray/triangle test that finds its
# surface (45) and the free flight and interaction arithmetic (55).
FLOP_PER_SEGMENT = 100.0
BYTES_PER_TRIANGLE = 36.0


def work(case):
    if case["kind"] == "hits":
        n_tri = len(CYLINDERS) * case["n_theta"] * 22
        per_ray = 32 + 12 + (4 if case["regions"] else 0)
        return {"bytes": case["n"] * per_ray + n_tri * BYTES_PER_TRIANGLE, "flops": case["n"] * 45.0}
    if case["kind"] == "batch":
        seg = (1.7, 2.0, 3.0)
        items = W.batch_instances(lo=case["lo"], hi=case["hi"])
        hist = sum(n * seg[s] for _, s, n, _ in items)
        n_inst, n_tri = len(items), 384
    else:
        n_inst = 1 if case["kind"] in ("run", "noalloc") else len(_instances(case))
        hist = n_inst * case["n"] * SETUPS[case["det"]][2]
        n_tri = 192 if case["det"] == "bare" else 157 * _detector(case).n_theta
    table = 4 * 3 * W.TABLE_N_GRID * 4
    return {"bytes": n_inst * W.N_BINS * 4 + n_tri * BYTES_PER_TRIANGLE + table, "flops": hist * FLOP_PER_SEGMENT}


def exact(case, seed):
    """The distances of a hits case from a brute-force search in 64 bits.  A transport
    run has no value in closed form, and its histories followed one by one in 64 bits
    take minutes."""
    if case["kind"] != "hits":
        return None
    xyz, tri, solid = _revolved_mesh(case["n_theta"])
    rays_np, reg = _rays(case, seed)
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    v = torch.from_numpy(xyz).double().to(dev)[torch.from_numpy(tri).long().to(dev)]
    rays = torch.from_numpy(rays_np[:, :7]).double().to(dev)
    out = torch.full((case["n"],), float("inf"), dtype=torch.float64, device=dev)
    solid = torch.from_numpy(solid).to(dev)
    # a ray of the world meets the can first; one of the active crystal its own surface
    groups = [(rays_np[:, 2] > 0, solid == 0), (rays_np[:, 2] <= 0, solid == len(CYLINDERS) - 1)]
    for who, tris in groups:
        idx = torch.from_numpy(np.nonzero(who)[0]).to(dev)
        a, b, c = (v[tris][:, k] for k in range(3))
        e1, e2 = b - a, c - a
        nrm = torch.linalg.cross(e1, e2)
        step = max(1, 20_000_000 // max(len(a), 1))
        for i in range(0, len(idx), step):
            sel = idx[i:i + step]
            o, d = rays[sel, 0:3], rays[sel, 4:7]
            # Moeller-Trumbore with the triple products taken as matrix products:
            # det = -d.n, u det = d.(e2 x (o-a)), v det = -d.(e1 x (o-a)), t det = n.(o-a)
            det = -(d @ nrm.T)
            m = torch.linalg.cross(o, d)
            u = m @ e2.T + d @ torch.linalg.cross(a, e2).T
            w = -(m @ e1.T) - d @ torch.linalg.cross(a, e1).T
            t = (o @ nrm.T - (a * nrm).sum(1)) / det
            u, w = u / det, w / det
            ok = (u >= -1e-12) & (w >= -1e-12) & (u + w <= 1.0 + 1e-12) & (t > 0)
            out[sel] = torch.where(ok, t, torch.full_like(t, float("inf"))).amin(1)
    return out, None, None
