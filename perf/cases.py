"""Performance cases: what a user of this engine has it do, each through its public entry points.

Three groups. Dose calculation: reset, transport, read the dose back (analytic beams and phase-space
records, photons and electrons, 5e4 to 1e8 histories, voxel-limited and voxel-crossing steps), a new
patient (materials, phantom, source, transport, dose) and the allocation-free call. Batched beamlets:
a new plan from its definition to the sparse dose-influence matrix, and the same plan run again. Dose
maps: merging a raw tally of another rank or checkpoint, the denoiser's inference alone and behind a
transport run, and its gradients. Phantoms, beams and history counts are those of the repository's
workloads (water 61x61x60, slab and half-slab 120^3, CT-like grids, 128^3 denoiser grids, 512-beamlet
recipe) or of their ranges.

Everything is made from the seed: phantom inserts, beam angles, records, tallies, dose maps, and the
transport's random streams. Transport has no value in 64 bits that single histories could be held to
(the tally is a sum of random samples), so exact() covers the dose maps only.
"""
import math
from statistics import NormalDist
from types import SimpleNamespace

import numpy as np
import torch
import torch.nn.functional as F

WEIGHTS = "paper_1503_01722_gb300/weights/unet_128.npy"
TALLY_SCALE = 2.0 ** 28

# compositions (Z, mass fraction), mean excitation energy (eV), nominal density (g/cm^3)
A_MASS = {1: 1.008, 6: 12.011, 7: 14.007, 8: 15.999, 11: 22.990, 12: 24.305, 15: 30.974, 16: 32.06,
          17: 35.45, 19: 39.098, 20: 40.078}
TISSUES = (
    (((1, 0.111894), (8, 0.888106)), 75.0, 1.0),
    (((1, 0.0472), (6, 0.1443), (7, 0.0420), (8, 0.4462), (12, 0.0022), (15, 0.1050), (16, 0.0031), (20, 0.2100)),
     106.4, 1.85),
    (((1, 0.1013), (6, 0.1023), (7, 0.0287), (8, 0.7571), (11, 0.0018), (15, 0.0008), (16, 0.0023), (17, 0.0027),
      (19, 0.0020)), 75.3, 0.26),
    (((1, 0.114), (6, 0.598), (7, 0.007), (8, 0.278), (11, 0.001), (16, 0.001), (17, 0.001)), 63.2, 0.95),
    (((1, 0.102), (6, 0.143), (7, 0.034), (8, 0.710), (11, 0.001), (15, 0.002), (16, 0.003), (17, 0.001),
      (19, 0.004)), 75.3, 1.05),
)


def listed():
    return [
        # the smallest call: 15 MeV electrons on the homogeneous water phantom at 0.5 cm, dose on the host
        {"name": "electron_water_61_5e4", "kind": "beam", "particle": "electron", "histories": 50_000, "nx": 61,
         "ny": 61, "nz": 60, "voxel": 0.5, "phantom": "water", "field": 10.0, "ssd": 0.0, "batches": 10,
         "cross": False, "host": True},
        # the headline workload: 6 MV photons on the slab phantom, dose on the host
        {"name": "photon_slab_120_1e8", "kind": "beam", "particle": "photon", "histories": 100_000_000, "nx": 120,
         "ny": 120, "nz": 120, "voxel": 0.25, "phantom": "slab", "field": 10.0, "ssd": 100.0, "batches": 10,
         "cross": False, "host": True},
        # electron beam at production size, dose kept on the device for what follows
        {"name": "electron_half_slab_120_1e7", "kind": "beam", "particle": "electron", "histories": 10_000_000,
         "nx": 120, "ny": 120, "nz": 120, "voxel": 0.25, "phantom": "half_slab", "field": 10.0, "ssd": 100.0,
         "batches": 10, "cross": False, "host": False},
        # linac phase space: photons with contaminant electrons and positrons, each record used about twice
        {"name": "phase_space_slab_120_2e6", "kind": "phase_space", "records": 1_000_000, "histories": 2_000_000,
         "nx": 120, "ny": 120, "nz": 120, "voxel": 0.25, "phantom": "slab", "field": 10.0, "batches": 10},
        # a new patient: tissue set, CT grid, beam, one run at a few percent of statistical error, dose on the host
        {"name": "new_patient_128_1e6", "kind": "patient", "particle": "photon", "histories": 1_000_000, "nx": 128,
         "ny": 128, "nz": 128, "voxel": 0.25, "materials": 5, "field": 8.0},
        # a planning host that forbids allocation: small electron run through the allocation-free call
        {"name": "noalloc_electron_61_2e5", "kind": "noalloc", "particle": "electron", "histories": 200_000,
         "nx": 61, "ny": 61, "nz": 60, "voxel": 0.5, "phantom": "water", "field": 10.0, "ssd": 0.0},
        # dose-influence matrix of a small plan, from the beamlet list to the sparse matrix on the host
        {"name": "beamlets_new_plan_64", "kind": "beamlets", "beamlets": 64, "log10_mean": 5.0, "nx": 128, "ny": 128,
         "nz": 96, "voxel": 0.25, "new_plan": True},
        # beamlets on the full CT grid, run again on tables and graph that are already there
        {"name": "beamlets_ct_192_again", "kind": "beamlets", "beamlets": 192, "log10_mean": 5.0, "nx": 256,
         "ny": 256, "nz": 128, "voxel": 0.2, "new_plan": False},
        # dose from a summed raw tally: what a rank does after the all-reduce, or a resumed run
        {"name": "merge_tally_120_b10", "kind": "merge", "nx": 120, "ny": 120, "nz": 120, "voxel": 0.25,
         "batches": 10, "log10_histories": 8.0},
        # the trained denoiser alone, on a dose map that is on the device
        {"name": "denoiser_forward_128", "kind": "forward", "nx": 128, "ny": 128, "nz": 128, "sigma": True},
        # the denoised dose calculation: a short run, then the network with its plain fallback
        {"name": "denoised_dose_128_1e6", "kind": "denoise", "particle": "photon", "histories": 1_280_000, "nx": 128,
         "ny": 128, "nz": 128, "voxel": 0.25, "field": 8.0},
        # the denoiser's loss and gradients on one training pair (a data-parallel step before its all-reduce)
        {"name": "denoiser_gradients_128", "kind": "gradients", "nx": 128, "ny": 128, "nz": 128, "sigma": True},
    ]


def log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["beam", "beam", "beam", "beam", "phase_space", "patient", "noalloc", "beamlets", "merge",
                       "forward", "denoise", "gradients"])
    grid = {k: rng.randint(24, 150) for k in ("nx", "ny", "nz")}
    c8 = {k: 8 * rng.randint(4, 16) for k in ("nx", "ny", "nz")}
    particle = rng.choice(["photon", "electron"])
    voxel = round(log_uniform(rng, 0.1, 0.5), 3)
    if kind == "beam":
        top = 2e7 if particle == "photon" else 2e6
        return {"kind": kind, "particle": particle, "histories": int(log_uniform(rng, 1e4, top)), **grid,
                "voxel": voxel, "phantom": rng.choice(["water", "slab", "half_slab", "ct"]),
                "field": round(rng.uniform(2.0, 20.0), 2), "ssd": rng.choice([0.0, 100.0]),
                "batches": rng.choice([5, 10, 10, 20]), "cross": rng.random() < 0.2, "host": rng.random() < 0.5}
    if kind == "phase_space":
        return {"kind": kind, "records": int(log_uniform(rng, 1e4, 2e6)), "histories": int(log_uniform(rng, 1e4, 5e6)),
                **grid, "voxel": voxel, "phantom": rng.choice(["water", "slab", "half_slab", "ct"]),
                "field": round(rng.uniform(2.0, 20.0), 2), "batches": rng.choice([5, 10, 10, 20])}
    if kind == "patient":
        return {"kind": kind, "particle": particle, "histories": int(log_uniform(rng, 1e4, 2e6)), **grid,
                "voxel": voxel, "materials": rng.randint(1, 5), "field": round(rng.uniform(2.0, 20.0), 2)}
    if kind == "noalloc":
        return {"kind": kind, "particle": particle, "histories": int(log_uniform(rng, 1e4, 1e6)), **grid,
                "voxel": voxel, "phantom": rng.choice(["water", "slab", "half_slab"]),
                "field": round(rng.uniform(2.0, 20.0), 2), "ssd": rng.choice([0.0, 100.0])}
    if kind == "beamlets":
        return {"kind": kind, "beamlets": int(log_uniform(rng, 4, 128)), "log10_mean": round(rng.uniform(4.0, 5.0), 2),
                **{k: rng.randint(48, 150) for k in ("nx", "ny", "nz")}, "voxel": round(rng.uniform(0.2, 0.4), 3),
                "new_plan": rng.random() < 0.5}
    if kind == "merge":
        return {"kind": kind, **grid, "voxel": voxel, "batches": rng.choice([1, 5, 10, 20]),
                "log10_histories": round(rng.uniform(5.0, 10.0), 2)}
    if kind == "denoise":
        return {"kind": kind, "particle": particle, "histories": int(log_uniform(rng, 1e5, 2e6)), **c8, "voxel": 0.25,
                "field": round(rng.uniform(2.0, 20.0), 2)}
    return {"kind": kind, **c8, "sigma": rng.random() < 0.7}


# ---- inputs ----------------------------------------------------------------------------------
def generator(seed, device="cuda"):
    g = torch.Generator(device=device)
    g.manual_seed(int(seed))
    return g


def axes(case, v):
    """Voxel centres (cm), shaped to broadcast over (nz, ny, nx)."""
    n = (case["nz"], case["ny"], case["nx"])
    z, y, x = ((torch.arange(k, device="cuda", dtype=torch.float32) + 0.5) * v for k in n)
    return n, z[:, None, None], y[None, :, None], x[None, None, :]


def ct_density(case, v, g):
    """A body ellipsoid of water with eight random inserts of density 0.2 to 1.9 g/cm^3, air around it."""
    n, z, y, x = axes(case, v)
    L = [n[2] * v, n[1] * v, n[0] * v]
    body = (((x - L[0] / 2) / (0.45 * L[0])) ** 2 + ((y - L[1] / 2) / (0.35 * L[1])) ** 2 +
            ((z - L[2] / 2) / (0.48 * L[2])) ** 2) <= 1
    d = torch.where(body, 1.0, 0.0012)
    u = torch.rand((8, 7), generator=g, device="cuda").tolist()
    for a in u:
        c = [(0.3 + 0.4 * a[0]) * L[0], (0.35 + 0.3 * a[1]) * L[1], (0.2 + 0.6 * a[2]) * L[2]]
        r = [(0.04 + 0.08 * a[3]) * L[0], (0.04 + 0.06 * a[4]) * L[1], (0.05 + 0.15 * a[5]) * L[2]]
        sel = (((x - c[0]) / r[0]) ** 2 + ((y - c[1]) / r[1]) ** 2 + ((z - c[2]) / r[2]) ** 2) <= 1
        d = torch.where(sel & body, 0.2 + 1.7 * a[6], d)
    return d, body


def ct_phantom(case, v, g):
    """Density, and water / bone / lung by density thresholds."""
    d, body = ct_density(case, v, g)
    m = torch.where(d < 0.6, 2, torch.where(d > 1.3, 1, 0))
    m = torch.where(body, m, 0).to(torch.uint8)
    return d.float().contiguous(), m.contiguous()


def phantom(case, g):
    """(density, material) on the device: water, layers, half layers or a CT-like body."""
    v, kind = case["voxel"], case["phantom"]
    if kind == "ct":
        return ct_phantom(case, v, g)
    n, z, y, x = axes(case, v)
    m = torch.zeros(n, dtype=torch.uint8, device="cuda")
    if kind == "slab":
        m = torch.where((z >= 3.0) & (z < 5.0), 1, torch.where((z >= 5.0) & (z < 12.0), 2, 0)).expand(n)
    elif kind == "half_slab":
        layer = (z >= 3.0) & (z < 10.0)
        m = torch.where(layer, torch.where(x < n[2] * v / 2, 1, 2), 0).expand(n)
    d = torch.tensor([1.0, 1.85, 0.26], device="cuda")[m.long()]
    return d.contiguous(), m.to(torch.uint8).contiguous()


def spectrum_6mv():
    """24 bins of the closed-form shape ((6 - E)/E)(1 - exp(-(E/1.3)^2)) on 0.25 to 6 MeV."""
    edges = np.linspace(0.25, 6.0, 25)
    e = edges[:-1, None] + (edges[1] - edges[0]) * (np.arange(64) + 0.5) / 64
    w = (((6.0 - e) / e) * (1.0 - np.exp(-(e / 1.3) ** 2))).sum(1)
    return edges.astype(np.float32), (w / w.sum()).astype(np.float32)


def spectrum(particle):
    if particle == "photon":
        return spectrum_6mv()
    return np.array([15.0, 15.0], np.float32), np.array([1.0], np.float32)


def beam(case, ssd):
    """Normal to the entrance face z = 0, centred on it."""
    v = case["voxel"]
    e, w = spectrum(case["particle"])
    return SimpleNamespace(particle=0 if case["particle"] == "photon" else 1, edges=e, weights=w,
                           field=(case["field"], case["field"]), ssd=ssd,
                           iso=(case["nx"] * v / 2, case["ny"] * v / 2, 0.0), direction=(0.0, 0.0, 1.0))


def gantry_beam(case, rng):
    """Through the phantom's centre at a random angle about y, source at 100 cm."""
    v, th = case["voxel"], rng.uniform(0.0, 2.0 * math.pi)
    b = beam(case, 100.0)
    b.iso = (case["nx"] * v / 2, case["ny"] * v / 2, case["nz"] * v / 2)
    b.direction = (math.sin(th), 0.0, math.cos(th))
    return b


def phase_space(case, rng):
    """Records above the entrance face from a point source at 100 cm with 0.5 degree blur: 94 % photons of
    the 6 MV spectrum, 5 % electrons, 1 % positrons."""
    n, v, f = case["records"], case["voxel"], case["field"]
    c = np.array([case["nx"] * v / 2, case["ny"] * v / 2, -100.0])
    P = np.zeros((n, 3))
    P[:, 0] = c[0] + rng.uniform(-0.5, 0.5, n) * f
    P[:, 1] = c[1] + rng.uniform(-0.5, 0.5, n) * f
    d = P - c
    d /= np.linalg.norm(d, axis=1, keepdims=True)
    d += rng.normal(0.0, math.radians(0.5), (n, 3))
    X = c + ((-2.0 - c[2]) / d[:, 2])[:, None] * d
    edges, w = spectrum_6mv()
    k = rng.random(n)
    typ = np.where(k < 0.01, 2, np.where(k < 0.06, 1, 0)).astype(np.int32)
    E = edges[rng.choice(24, size=n, p=w / w.sum(dtype=np.float64))] + rng.random(n) * (edges[1] - edges[0])
    E = np.where(typ == 1, rng.uniform(0.5, 6.0, n), np.where(typ == 2, rng.uniform(0.5, 4.0, n), E))
    rec = np.zeros(n, np.dtype([(a, "<f4") for a in "xyzuvwE"] + [("type", "<i4")]))
    for i, a in enumerate("xyz"):
        rec[a] = X[:, i]
    for i, a in enumerate("uvw"):
        rec[a] = d[:, i]
    rec["E"], rec["type"] = E, typ
    return rec


def beamlet_histories(case):
    """Lognormal over the plan (sd 0.5 in log10, 1e4 to 1e6): the distribution's own quantiles, in beamlet order."""
    n = case["beamlets"]
    q = [NormalDist().inv_cdf((i + 0.5) / n) for i in range(n)]
    return [int(min(max(round(10.0 ** (case["log10_mean"] + 0.5 * z)), 10_000), 1_000_000)) for z in q]


def beamlet_room(case):
    """Entries that a plan's matrix has room for: a beamlet's footprint grows with its histories, up to the grid."""
    nvox = case["nx"] * case["ny"] * case["nz"]
    return sum(int(min(nvox, 24 * n ** 0.85)) for n in beamlet_histories(case))


def beamlet_list(case, rng):
    """0.5 x 0.5 cm^2 at random gantry angles about the centre, offsets up to 4 cm."""
    v = case["voxel"]
    c = np.array([case["nx"] * v / 2, case["ny"] * v / 2, case["nz"] * v / 2])
    out = []
    for n in beamlet_histories(case):
        th = rng.uniform(0.0, 2.0 * math.pi)
        a, b = rng.uniform(-4.0, 4.0, 2)
        iso = c + a * np.array([math.cos(th), 0.0, -math.sin(th)]) + b * np.array([0.0, 1.0, 0.0])
        out.append({"field": (0.5, 0.5), "ssd": 100.0, "iso": tuple(iso), "direction": (math.sin(th), 0.0, math.cos(th)),
                    "n_histories": n})
    return out


def dose_maps(case, seed):
    """A noisy dose map with its batch sigma, the density and a smooth dose to train towards."""
    g = generator(seed)
    v = 0.25
    dens, _ = ct_density(case, v, g)
    n, z, y, x = axes(case, v)
    u = torch.rand(4, generator=g, device="cuda").tolist()
    fx, fy = 2.0 + 10.0 * u[0], 2.0 + 10.0 * u[1]
    cx, cy = n[2] * v * (0.4 + 0.2 * u[2]), n[1] * v * (0.4 + 0.2 * u[3])
    depth = torch.cumsum(dens, 0) * v
    edge = torch.sigmoid((fx / 2 - (x - cx).abs()) / 0.3) * torch.sigmoid((fy / 2 - (y - cy).abs()) / 0.3)
    true = 1e-3 * (edge * (1.0 - 0.7 * torch.exp(-depth / 0.5)) + 0.01) * torch.exp(-0.045 * depth)
    sigma = (0.04 * 1e-3 * (true / 1e-3).sqrt()).contiguous()
    # the map to learn: the smooth dose of a machine whose output is a fifth lower
    target = 0.8 * true
    noisy = (true + sigma * torch.randn(n, generator=g, device="cuda")).clamp_min(0.0).contiguous()
    return noisy, sigma, dens.float().contiguous(), target.float().contiguous()


def raw_tally(case, seed):
    """A summed tally in fixed-point units: a depth-dose with Poisson-like noise in every batch, and the density."""
    g = generator(seed)
    v, B, N = case["voxel"], case["batches"], int(10 ** case["log10_histories"])
    dens, _ = ct_density(case, v, g)
    n, z, y, x = axes(case, v)
    r = torch.exp(-((x - n[2] * v / 2) ** 2 + (y - n[1] * v / 2) ** 2) / 20.0) + 1e-3
    mean = 2e-7 * r * torch.exp(-0.05 * z) * TALLY_SCALE * (N / B)
    t = torch.empty((B,) + n, dtype=torch.int64, device="cuda")
    for b in range(B):
        t[b] = (mean * (1.0 + 0.05 * torch.randn(n, generator=g, device="cuda"))).clamp_min(0.0).to(torch.int64)
    dens = torch.where(torch.rand(n, generator=g, device="cuda") < 0.01, 0.0, dens).contiguous()
    return t, dens, N


# ---- the calls ---------------------------------------------------------------------------------
def prepare(case, seed):
    from paper_1503_01722_gb300 import ocmc
    kind, s = case["kind"], SimpleNamespace(kind=case["kind"], case=case, ocmc=ocmc, seed=int(seed) + 1)
    g, rng = generator(seed), np.random.default_rng(int(seed))
    shape = (case["nz"], case["ny"], case["nx"])
    if kind in ("beam", "phase_space"):
        kw = {"n_batches": case["batches"]}
        if case.get("cross"):
            kw["flags"] = ocmc.FLAG_CROSS_VOXELS
        s.e = ocmc.Engine(0, **kw)
        d, m = (t.cpu().numpy() for t in phantom(case, g))
        s.e.create_phantom(density=d, material=m, voxel=(case["voxel"],) * 3)
        if kind == "beam":
            s.e.set_source(beam(case, case["ssd"]))
        else:
            s.e.set_phase_space(phase_space(case, rng))
        s.host = case.get("host", False)
        s.out = None if s.host else (torch.empty(shape, device="cuda"), torch.empty(shape, device="cuda"))
    elif kind == "patient":
        d, body = ct_density(case, case["voxel"], g)
        d, k = d.float().contiguous(), case["materials"]
        # materials by density: lung, adipose, muscle, bone around water, as many as are defined
        m = torch.zeros(shape, dtype=torch.uint8, device="cuda")
        for lo, hi, t in ((1.3, 30.0, 1), (0.0, 0.6, 2), (0.6, 0.97, 3), (1.02, 1.3, 4)):
            if t < k:
                m = torch.where(body & (d > lo) & (d <= hi), t, m).to(torch.uint8)
        s.density, s.material = d.cpu().numpy(), m.cpu().numpy()
        s.tissues = [{"Z": [z for z, _ in zw], "A": [A_MASS[z] for z, _ in zw], "w": [w for _, w in zw], "I": I,
                      "density": rho} for zw, I, rho in TISSUES[:k]]
        s.beam = gantry_beam(case, rng)
        s.e = ocmc.Engine(0)
    elif kind == "noalloc":
        s.density, s.material = phantom(case, g)
        s.beam = beam(case, case["ssd"])
        s.tally = torch.zeros((10,) + shape, dtype=torch.int64, device="cuda")
    elif kind == "beamlets":
        s.e = ocmc.Engine(0)
        d, m = (t.cpu().numpy() for t in ct_phantom(case, case["voxel"], g))
        s.e.create_phantom(density=d, material=m, voxel=(case["voxel"],) * 3)
        s.list, s.spectrum = beamlet_list(case, rng), spectrum_6mv()
        if not case["new_plan"]:
            s.e.set_beamlets(0, *s.spectrum, s.list)
        # the matrix by columns: a program knows its plans' size and keeps the arrays
        room = beamlet_room(case)
        s.indptr = np.zeros(case["beamlets"] + 1, np.int64)
        s.indices, s.data = np.zeros(room, np.int32), np.zeros(room, np.float32)
    elif kind == "merge":
        s.tally, dens, s.N = raw_tally(case, seed)
        s.e = ocmc.Engine(0, n_batches=case["batches"])
        s.e.create_phantom(density=dens.cpu().numpy(), material=np.zeros(shape, np.uint8), voxel=(case["voxel"],) * 3)
        s.out = (torch.empty(shape, device="cuda"), torch.empty(shape, device="cuda"))
    elif kind in ("forward", "gradients"):
        s.dose, s.sigma, s.density, s.target = dose_maps(case, seed)
        s.sigma = s.sigma if case["sigma"] else None
        s.net = ocmc.UNet(shape)
        s.net.set_params(np.load(WEIGHTS))
        s.out = torch.empty(shape, device="cuda")
    else:
        s.e = ocmc.Engine(0)
        d, m = (t.cpu().numpy() for t in ct_phantom(case, case["voxel"], g))
        s.e.create_phantom(density=d, material=m, voxel=(case["voxel"],) * 3)
        s.e.set_source(gantry_beam(case, rng))
        s.net = ocmc.UNet(shape)
        s.net.set_params(np.load(WEIGHTS))
        s.out, s.flag = torch.empty(shape, device="cuda"), torch.empty(shape, device="cuda")
    torch.cuda.synchronize()
    return s


def run(s):
    kind, c = s.kind, s.case
    if kind in ("beam", "phase_space"):
        s.e.reset()
        s.e.run(c["histories"], seed=s.seed)
        return s.e.dose() if s.out is None else s.e.dose(out=s.out)
    if kind == "patient":
        s.e.set_materials(s.tissues)
        s.e.create_phantom(density=s.density, material=s.material, voxel=(c["voxel"],) * 3)
        s.e.set_source(s.beam)
        s.e.run(c["histories"], seed=s.seed)
        return s.e.dose()
    if kind == "noalloc":
        s.tally.zero_()
        s.ocmc.run_noalloc(s.density, s.material, (c["voxel"],) * 3, s.beam, s.tally, 0, c["histories"],
                           c["histories"], seed=s.seed)
        return s.tally
    if kind == "beamlets":
        if c["new_plan"]:
            s.e.set_beamlets(0, *s.spectrum, s.list)
        s.e.run_beamlets(seed=s.seed)
        at = 0
        for b, (i, d) in enumerate(s.e.beamlet_doses()):
            s.indices[at:at + len(i)], s.data[at:at + len(i)] = i, d
            at += len(i)
            s.indptr[b + 1] = at
        return {"indptr": s.indptr, "indices": s.indices, "data": s.data}
    if kind == "merge":
        s.e.reset()
        s.e.add_raw_tally(s.tally, 0, s.N)
        return s.e.dose(out=s.out)
    if kind == "forward":
        return s.net.forward(s.dose, s.density, s.out, sigma=s.sigma)
    if kind == "gradients":
        loss = s.net.train_step(s.dose, s.density, s.target, 0.0, sigma=s.sigma)
        return {"loss": loss, "gradients": s.net.params(grads=True)}
    s.e.reset()
    s.e.run(c["histories"], seed=s.seed)
    return s.ocmc.denoise(s.e, s.net, 4.0, s.out, s.flag)


# ---- what a pass cannot do without ----------------------------------------------------------------
def network_flops(nvox):
    """Multiply-adds times two of one forward pass: 27-tap layers at their grid, 8-tap layers at the coarse one."""
    conv = [(16, 16, 1), (16, 16, 1), (32, 32, 8), (32, 32, 8), (64, 64, 64), (64, 64, 64), (128, 128, 512),
            (128, 128, 512), (128, 64, 64), (64, 64, 64), (64, 32, 8), (32, 32, 8), (32, 16, 1), (16, 16, 1)]
    half = [(16, 32, 8), (32, 64, 64), (64, 128, 512), (128, 64, 512), (64, 32, 64), (32, 16, 8)]
    return 2.0 * nvox * (sum(27 * a * b / f for a, b, f in conv) + sum(8 * a * b / f for a, b, f in half))


def work(case):
    kind = case["kind"]
    n = case["nx"] * case["ny"] * case["nz"]
    # about 34 particle steps a 6 MV photon history and 180 a 15 MeV electron history, about 300 operations each
    ops = {"photon": 34 * 300.0, "electron": 180 * 300.0}
    if kind in ("beam", "patient"):
        return {"bytes": 13.0 * n, "flops": case["histories"] * ops[case["particle"]]}
    if kind == "phase_space":
        return {"bytes": 13.0 * n + 32.0 * case["records"], "flops": case["histories"] * ops["photon"]}
    if kind == "noalloc":
        return {"bytes": 5.0 * n + 80.0 * n, "flops": case["histories"] * ops[case["particle"]]}
    if kind == "beamlets":
        # index and dose of each entry; about half of the room is filled
        return {"bytes": 5.0 * n + 4.0 * beamlet_room(case), "flops": sum(beamlet_histories(case)) * ops["photon"]}
    if kind == "merge":
        return {"bytes": n * (8.0 * case["batches"] + 12.0), "flops": n * (6.0 * case["batches"] + 6.0)}
    if kind == "forward":
        return {"bytes": n * (12.0 + 4.0 * case["sigma"]) + 7.1e6, "flops": network_flops(n)}
    if kind == "gradients":
        return {"bytes": n * (12.0 + 4.0 * case["sigma"]) + 14.2e6, "flops": 3.0 * network_flops(n)}
    return {"bytes": 13.0 * n + 7.1e6, "flops": network_flops(n) + case["histories"] * ops[case["particle"]]}


# ---- the same outputs in 64 bits -----------------------------------------------------------------
CHANNELS = (16, 32, 64, 128)


def architecture():
    """(kind, in, out) of the network's layers in the order of the flat parameter vector."""
    L, c = [], 16
    for l, C in enumerate(CHANNELS):
        L += [("conv", c, C), ("conv", C, C)]
        if l < 3:
            L.append(("down", C, CHANNELS[l + 1]))
            c = CHANNELS[l + 1]
    p = 128
    for C in (64, 32, 16):
        L += [("up", p, C), ("conv", 2 * C, C), ("conv", C, C)]
        p = C
    return L


def network(p, x):
    """The U-Net on x (1, 16, nz, ny, nx) with the flat parameters p: last feature map of 16 channels."""
    at, i, skip, L = 0, 0, [], architecture()

    def layer(x):
        nonlocal at, i
        k, a, b = L[i]
        t = 3 if k == "conv" else 2
        w = p[at:at + t ** 3 * a * b].reshape(t, t, t, a, b)
        bias = p[at + t ** 3 * a * b:at + t ** 3 * a * b + b]
        at, i = at + t ** 3 * a * b + b, i + 1
        if k == "conv":
            y = F.conv3d(x, w.permute(4, 3, 0, 1, 2), bias, padding=1)
        elif k == "down":
            y = F.conv3d(x, w.permute(4, 3, 0, 1, 2), bias, stride=2)
        else:
            y = F.conv_transpose3d(x, w.permute(3, 4, 0, 1, 2), bias, stride=2)
        return torch.relu(y)

    for l in range(4):
        x = layer(layer(x))
        if l < 3:
            skip.append(x)
            x = layer(x)
    for l in range(3):
        x = layer(layer(torch.cat([layer(x), skip.pop()], 1)))
    return x, at


def exact(case, seed):
    kind = case["kind"]
    if kind == "merge":
        t, dens, N = raw_tally(case, seed)
        B, v = case["batches"], case["voxel"]
        rho = dens.double()
        unit = TALLY_SCALE * float(np.float32(v)) ** 3 * rho
        n_b = [(N - b - 1) // B + 1 if N > b else 0 for b in range(B)]
        D = t.double().sum(0) / (unit * N)
        if B > 1:
            S = sum((t[b].double() / (unit * n_b[b]) - D) ** 2 for b in range(B))
            S = (S / (B * (B - 1))).sqrt()
        else:
            S = torch.zeros_like(D)
        zero = torch.zeros_like(D)
        return torch.where(rho > 0, D, zero), torch.where(rho > 0, S, zero)
    if kind not in ("forward", "gradients"):
        return None
    dose, sigma, dens, target = (a.double() for a in dose_maps(case, seed))
    p = torch.from_numpy(np.load(WEIGHTS)).cuda().double().requires_grad_(kind == "gradients")
    s = dose.max()
    x = torch.zeros((1, 16) + tuple(dose.shape), dtype=torch.float64, device="cuda")
    x[0, 0], x[0, 1] = dose / s, dens
    if case["sigma"]:
        x[0, 2] = sigma / s
    with torch.set_grad_enabled(kind == "gradients"):
        h, at = network(p, x)
        out = dose / s + (h[0] * p[at:at + 16, None, None, None]).sum(0) + p[at + 16]
        if kind == "forward":
            return out * s
        body = dens >= 0.1
        loss = (((out - target / s) ** 2) * body).sum() / body.sum()
        loss.backward()
    return {"loss": loss.detach(), "gradients": p.grad}
