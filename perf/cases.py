"""Performance cases of the two-beam FFT-BPM march, through the public entry points.

Each case is one call (or one burst of calls) that a user of the library
makes, at sizes of the project's own workloads (``inputs.py``, the tests and
the benchmark) or inside the ranges that the C ABI documents.  A case is a
dict of plain values; ``prepare`` builds what a user holds before the call
(inputs and a plan), ``run`` makes the call, ``exact`` gives the same outputs
from a plain complex128 march written with torch alone.
"""

import cmath
import math
import random

import numpy as np
import torch

from paper_2601_06340_gb300 import binding as bpm
from paper_2601_06340_gb300 import inputs

HC_EV_ANGSTROM = 12398.419843320026
E_REF_EV = 8000.0                        # the configured reflection: Si(220)-like at 8 keV
THETA_REF = math.radians(23.65)
CHI0 = complex(-1.51e-5, 3.5e-7)
CHIH = complex(-9.1e-6, 3.4e-7)
E_440_EV = 17450.0                       # the 3D example: Si(440)-like at 17.45 keV
THETA_440 = math.asin(HC_EV_ANGSTROM / E_440_EV * 1e-4 / (2.0 * 5.4309e-4 / math.sqrt(32.0)))
CHI0_440 = complex(-3.17e-6, 1.6e-8)
CHIH_440 = complex(-1.45e-6, 1.2e-8)
VACUUM, BULK, SLAB, SLAB_AND_POLYGON, BOX = 0, 1, 2, 5, 6
NONE, BENT, DISLOCATION = 0, 2, 3
SPLITS = {"first": 0, "verlet": 1, "forest_ruth": 2}
# (a_i, b_i) of the splitting's stages: propagate a_i dz, then couple b_i dz
_T = 1.0 / (2.0 - 2.0 ** (1.0 / 3.0))
STAGES = {
    "first": [(1.0, 1.0)],
    "verlet": [(0.0, 0.5), (1.0, 0.5)],
    "forest_ruth": [(0.0, _T / 2), (_T, (1 - _T) / 2), (1 - 2 * _T, (1 - _T) / 2), (_T, _T / 2)],
}


def march(name, geometry, nx, nz, rows=1, precision="fp32", split="first", record_every=0,
          api="device", dx_um=0.2, dz_um=0.1):
    c = dict(kind="march", geometry=geometry, nx=nx, nz=nz, rows=rows, precision=precision,
             split=split, record_every=record_every, api=api, dx_um=dx_um, dz_um=dz_um)
    return dict(c, name=name) if name else c


def listed():
    return [
        # Far-field image of an exit wave: one free-space step of metres, a
        # call made once per recorded image.  The smallest call: launches and
        # latency.
        march("far_field_2048", "far_field", 2048, 1, dz_um=2.0e6),
        # The perfect Laue crystal of the paper's first example, one solve
        # through the blocking host call with records and band powers.
        march("laue_1024_host", "laue", 1024, 2000, record_every=100, api="host", dx_um=0.4,
              dz_um=0.05),
        # The same solve in double precision, as the reference result that
        # single-precision solves are checked against.
        march("laue_1024_fp64", "laue", 1024, 2000, precision="fp64", record_every=100,
              api="host", dx_um=0.4, dz_um=0.05),
        # A short double-precision scan over incidence angles.
        march("rocking_24x2048_fp64", "rocking", 2048, 150, rows=24, precision="fp64",
              dx_um=0.4, dz_um=0.05),
        # The bent Bragg crystal on device buffers with records: the
        # benchmark's headline march, its first half (4000 of 8000 steps).
        march("bragg_bent_4096", "bragg_bent", 4096, 4000, record_every=100),
        # Dislocation in a polygon-shaped asymmetric crystal (per-cell strain
        # stream), half of the configured 12000 steps.
        march("asym_8192", "asym", 8192, 6000, record_every=200, dx_um=0.1, dz_um=0.05),
        # The largest grid, a bent Laue crystal.
        march("laue_bent_16384", "laue_bent", 16384, 2000, dx_um=0.1, dz_um=0.05),
        # Second-order splitting, which halves the step error, on a bent
        # Bragg crystal of ordinary size.
        march("verlet_2048", "bragg_bent", 2048, 2001, split="verlet", record_every=200),
        # A rocking curve: an odd number of angles through one Laue slab,
        # reflectivities from the band powers.
        march("rocking_101x2048", "rocking", 2048, 1000, rows=101, dx_um=0.4, dz_um=0.05),
        # A pulse: 256 photon energies through one bent Laue crystal, then
        # the field over time.
        dict(march(None, "pulse", 4096, 1000, rows=256, dx_um=0.1, dz_um=0.05),
             name="pulse_256x4096"),
        # Both transverse coordinates: the 10 um cube with a dislocation.
        dict(name="cube_512x256", kind="cube", nx=512, ny=256, nz=300, rows=1, split="first",
             step_um=0.05),
        # A burst of independent requests of mixed size, step count and
        # geometry served by the continuous-batching server.
        dict(name="serve_mix_24", kind="serve", requests=24, nz_min=500, nz_max=4000, mix=1),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng: random.Random):
    """Another case of the listed ranges: any grid size, odd step, row and record counts."""
    what = rng.choice(["far", "single", "single", "single", "fp64", "rows", "rows", "pulse",
                       "cube", "serve"])
    if what == "far":
        return march(None, "far_field", 2 ** rng.randint(6, 14), 1, rows=_log_int(rng, 1, 32),
                     dz_um=rng.uniform(1.0e6, 4.0e6))
    if what == "single":
        split = rng.choice(["first", "first", "verlet", "forest_ruth"])
        nx = 2 ** rng.randint(6, 13 if split == "forest_ruth" else 14)
        geometry = rng.choice(["bragg_bent", "laue", "laue_bent", "asym"])
        return march(None, geometry, nx, _log_int(rng, 50, 3000), split=split,
                     record_every=rng.choice([0, 0, rng.randint(40, 400)]),
                     api=rng.choice(["device", "device", "host"]),
                     dx_um=rng.uniform(0.1, 0.2), dz_um=rng.uniform(0.05, 0.1))
    if what == "fp64":
        nx = 2 ** rng.randint(6, 14)
        rows = _log_int(rng, 1, max(1, min(64, 262144 // nx)))
        return march(None, rng.choice(["laue", "laue_bent", "rocking", "bragg_bent"]), nx,
                     _log_int(rng, 30, 600), rows=rows, precision="fp64",
                     split=rng.choice(["first", "first", "verlet", "forest_ruth"]),
                     record_every=rng.choice([0, rng.randint(10, 100)]),
                     api=rng.choice(["device", "host"]),
                     dx_um=rng.uniform(0.1, 0.4), dz_um=rng.uniform(0.05, 0.1))
    if what == "rows":
        nx = 2 ** rng.randint(8, 13)
        rows = _log_int(rng, 2, min(256, 1048576 // nx))
        nz = min(_log_int(rng, 50, 3000), 900_000_000 // (nx * rows))
        return march(None, rng.choice(["rocking", "laue_bent"]), nx, nz, rows=rows,
                     split=rng.choice(["first", "first", "first", "verlet"]),
                     dx_um=rng.uniform(0.1, 0.4), dz_um=rng.uniform(0.05, 0.1))
    if what == "pulse":
        nx = 2 ** rng.randint(9, 12)
        return march(None, "pulse", nx, _log_int(rng, 50, 900), rows=2 ** rng.randint(3, 8),
                     dx_um=0.1, dz_um=0.05)
    if what == "cube":
        return dict(kind="cube", nx=2 ** rng.randint(8, 10), ny=2 ** rng.randint(8, 9),
                    nz=_log_int(rng, 30, 250), rows=rng.choice([1, 1, 2]),
                    split=rng.choice(["first", "first", "verlet"]),
                    step_um=rng.uniform(0.04, 0.06))
    return dict(kind="serve", requests=rng.randint(4, 24), nz_min=200,
                nz_max=_log_int(rng, 500, 4000), mix=rng.randint(2, 1 << 20))


# ---- inputs: numbers and arrays from the case and the seed alone --------------


def _gauss(x, centre, fwhm):
    return np.exp(-2.0 * math.log(2.0) * ((x - centre) / fwhm) ** 2)


def _polygon(rs, centre, extent):
    nv = int(rs.randint(5, 9))
    ang = np.sort(rs.uniform(0.0, 2.0 * math.pi, nv))
    rad = rs.uniform(0.5, 1.0, nv) * extent / 2.0
    return np.stack([centre[0] + rad * np.cos(ang), centre[1] + rad * np.sin(ang)], axis=1)


def _setup(case, seed):
    """The problem as plain numbers: grid, energies, crystal, strain, incident field."""
    rs = np.random.RandomState(seed % (1 << 31))
    nx, nz, rows = case["nx"], case["nz"], case["rows"]
    dx, dz, geometry = case["dx_um"], case["dz_um"], case["geometry"]
    width, length = nx * dx, nz * dz
    x0 = -0.5 * width
    x = x0 + np.arange(nx) * dx
    s, c = math.sin(THETA_REF), math.cos(THETA_REF)
    tan_t = s / c
    k = 2.0 * math.pi / (HC_EV_ANGSTROM / E_REF_EV * 1e-4)
    p = dict(nx=nx, nz=nz, rows=rows, dx=dx, dz=dz, x0=x0, e_ref=E_REF_EV, theta=THETA_REF,
             chi0=CHI0, chih=CHIH, energies=np.full(rows, E_REF_EV), ny=1)
    # surfaces half a cell off the grid: no cell centre lies on a face
    off = 0.5 * dx
    thick = min(300.0, 0.25 * width) + 0.25 * dx
    fwhm = min(50.0, 0.1 * width) * rs.uniform(0.8, 1.2)
    slab = dict(kind=SLAB, angle=0.0, thick=thick, surf=(off, 0.0))
    bent = (BENT, [1e6 * rs.uniform(0.5, 5.0), 0.28, 0.0, 0.5 * length])
    centre = max(-tan_t * 0.3 * length, 0.5 * x0) + 2.0 * dx * rs.uniform(-1, 1)
    strain, tilt = (NONE, [0.0] * 4), np.zeros(rows)
    amp = np.exp(2j * math.pi * rs.uniform(0.0, 1.0, rows))
    if geometry in ("laue", "laue_bent", "rocking", "pulse"):
        # a Laue slab that fills the march, the fan centred in the window
        slab = dict(kind=SLAB, angle=math.pi / 2, thick=length + dz, surf=(0.0, -0.25 * dz))
        centre = max(-0.5 * tan_t * length, 0.5 * x0) + 2.0 * dx * rs.uniform(-1, 1)
        if geometry != "laue" and (geometry != "rocking" or rs.uniform() < 0.5):
            strain = bent
    if geometry == "rocking":
        tilt = k * c * np.linspace(-50e-6, 50e-6, rows) + rs.uniform(-1, 1) * 1e-7 * k
        fwhm = min(200.0, 0.2 * width)
    elif geometry == "pulse":
        p["energies"] = 9000.0 - 5.0 + 10.0 * np.arange(rows) / rows
        amp = amp * np.exp(-((p["energies"] - 9000.0) ** 2) / (4.0 * 1.5 ** 2))
        s0 = s * E_REF_EV / 9000.0
        sj = s * E_REF_EV / p["energies"]
        tilt = (s0 - sj) * 2.0 * math.pi / (HC_EV_ANGSTROM / p["energies"] * 1e-4)
    elif geometry == "bragg_bent":
        strain = bent
    elif geometry == "asym":
        a = math.radians(rs.uniform(5.0, 30.0))
        n = (math.cos(a), math.sin(a))
        surf = (off, 0.5 * length)
        extent = max(40.0 * dx, min(300.0, 0.3 * width) * rs.uniform(0.5, 1.0))
        depth = min(20.0, 0.2 * extent)
        mid = (surf[0] + n[0] * extent / 2, surf[1] + n[1] * extent / 2)
        slab = dict(kind=SLAB_AND_POLYGON, angle=a, thick=300.0 + 0.25 * dx, surf=surf,
                    polygon=_polygon(rs, mid, extent))
        strain = (DISLOCATION, [3.84e-4, 0.28, surf[0] + n[0] * depth + 0.3 * dx,
                                surf[1] + n[1] * depth + 0.3 * dz])
    elif geometry == "far_field":
        slab = dict(kind=VACUUM, angle=0.0, thick=0.0, surf=(0.0, 0.0))
        p.update(chi0=0j, chih=0j)
    psi = np.zeros((rows, 2, nx), np.complex128)
    for r in range(rows):
        psi[r, 0] = amp[r] * _gauss(x, centre, fwhm / c) * np.exp(1j * tilt[r] * (x - centre))
    if geometry == "far_field":   # an exit wave has both bands
        psi[:, 1] = 0.7 * _gauss(x, -centre, fwhm / c)
    p.update(slab=slab, strain=strain, psi=psi)
    return p


def _setup_cube(case, seed):
    rs = np.random.RandomState(seed % (1 << 31))
    nx, ny, nz, d, rows = case["nx"], case["ny"], case["nz"], case["step_um"], case["rows"]
    cube = 200.0 * d
    x0, y0 = -0.42 * nx * d, -0.5 * ny * d
    s, c = math.sin(THETA_440), math.cos(THETA_440)
    x, y = x0 + np.arange(nx) * d, y0 + np.arange(ny) * d
    fwhm = 40.0 * d * rs.uniform(0.8, 1.2)
    xb = max(-s / c * min(0.75 * cube, 0.5 * nz * d), 0.5 * x0)
    psi = np.zeros((rows, 2, ny, nx), np.complex128)
    for r in range(rows):
        gx, gy = _gauss(x, xb + d * rs.uniform(-4, 4), fwhm / c), _gauss(y, d * rs.uniform(-4, 4), fwhm)
        psi[r, 0] = gy[:, None] * gx[None, :]
    q = 0.3 * d    # faces off the cell centres
    box = [-q, cube - q, -0.3 * ny * d - q, 0.3 * ny * d - q, min(0.25 * cube, 0.2 * nz * d) + q,
           1.25 * cube + q]
    strain = (DISLOCATION, [3.84e-4, 0.28, 0.5 * cube + 0.4 * d, min(0.75 * cube, 0.5 * nz * d) + 0.4 * d])
    return dict(nx=nx, ny=ny, nz=nz, rows=rows, dx=d, dy=d, dz=d, x0=x0, y0=y0, e_ref=E_440_EV,
                theta=THETA_440, chi0=CHI0_440, chih=CHIH_440,
                energies=E_440_EV + 2.0 * np.arange(rows),
                slab=dict(kind=BOX, box=box), strain=strain, psi=psi)


def _request_cases(case):
    """The burst's requests: sizes and step counts are the case's, not the seed's."""
    rng = random.Random(case["mix"])
    out = []
    for _ in range(case["requests"]):
        out.append(march(None, rng.choice(["bragg_bent", "laue_bent", "asym"]),
                         2 ** rng.randint(9, 14), rng.randint(case["nz_min"], case["nz_max"]),
                         api="host", dx_um=0.1, dz_um=0.05))
    return out


def _plan(case, p):
    """What a user's program builds: the workload and its plan."""
    s = p["slab"]
    if s["kind"] == BOX:
        crystal = dict(kind=BOX, box_um=s["box"])
    else:
        crystal = dict(kind=s["kind"], asym_angle_rad=s["angle"], thickness_um=s["thick"],
                       surf_x_um=s["surf"][0], surf_z_um=s["surf"][1])
        if "polygon" in s:
            crystal["polygon"] = s["polygon"]
    strain = dict(kind=p["strain"][0], params=p["strain"][1])
    common = ("case", p["nx"], p["nz"], p["dx"], p["dz"], p["x0"], p["energies"], p["e_ref"],
              p["theta"], p["chi0"], p["chih"], case.get("record_every", 0), crystal, strain,
              p["psi"])
    if p["ny"] > 1:
        wl = inputs.Workload3D(*common, ny=p["ny"], dy_um=p["dy"], y0_um=p["y0"])
    else:
        wl = inputs.Workload(*common)
    precision = bpm.BPM_FP64_PLAIN if case.get("precision") == "fp64" else bpm.BPM_FP32_FUSED
    return bpm.Plan(wl, precision, splitting=SPLITS[case.get("split", "first")])


def _host_outputs(psi, plan):
    """Result buffers of a host call: the exit field and, with records, those."""
    return bpm.MarchOutput(np.empty_like(psi),
                           np.zeros((psi.shape[0], plan.n_rec) + psi.shape[1:], plan.rec_dtype),
                           np.zeros((psi.shape[0], plan.n_rec + 1, 2)))


def prepare(case, seed):
    if case["kind"] == "serve":
        items = []
        for i, c in enumerate(_request_cases(case)):
            p = _setup(c, seed * 1000 + i)
            items.append((_plan(c, p), p["psi"], np.empty_like(p["psi"])))
        return dict(case=case, items=items)
    p = _setup_cube(case, seed) if case["kind"] == "cube" else _setup(case, seed)
    plan = _plan(case, p)
    st = dict(case=case, plan=plan)
    if case.get("api") == "host":
        st["psi"] = p["psi"]
        st["out"] = _host_outputs(p["psi"], plan)
        return st
    dtype = torch.complex128 if case.get("precision") == "fp64" else torch.complex64
    st["psi"] = torch.from_numpy(p["psi"]).to(device="cuda", dtype=dtype)
    st["out"] = torch.empty_like(st["psi"])
    shape = (p["rows"], plan.n_rec) + tuple(st["psi"].shape[1:])
    st["records"] = torch.zeros(shape, dtype=dtype, device="cuda") if plan.n_rec else None
    if case.get("geometry") == "rocking":
        st["powers"] = torch.zeros((p["rows"], plan.n_rec + 1, 2), dtype=torch.float64, device="cuda")
    if case.get("geometry") == "pulse":
        st["time"] = torch.empty((2, p["nx"], p["rows"]), dtype=dtype, device="cuda")
    return st


def run(st):
    case = st["case"]
    if case["kind"] == "serve":
        tickets = [bpm.bpm_submit(plan.handle, psi, out) for plan, psi, out in st["items"]]
        for t in tickets:
            bpm.bpm_poll(t, -1)
        # single-precision marches: kept as such
        return [out.astype(np.complex64) for _, _, out in st["items"]]
    plan = st["plan"]
    if case.get("api") == "host":
        out = plan.propagate(st["psi"], records=plan.n_rec > 0, out=st["out"])
        if case["precision"] == "fp64":
            return [out.psi, out.records, out.powers]
        return [out.psi.astype(np.complex64), out.records, out.powers.astype(np.float32)]
    stream = torch.cuda.current_stream().cuda_stream
    powers = st.get("powers")
    bpm.bpm_propagate_device(plan.handle, st["psi"], st["out"], st["records"], powers, 0,
                             case["nz"], stream)
    outs = [st["out"]]
    if st["records"] is not None:
        outs.append(st["records"])
    if powers is not None:   # the rocking curve, in the march's precision
        outs.append(powers if case["precision"] == "fp64" else powers.float())
    if "time" in st:
        bpm.bpm_omega_to_t_device(st["out"], st["time"], case["rows"], case["nx"],
                                  plan.precision, stream)
        outs.append(st["time"])
    return outs


def work(case):
    if case["kind"] == "serve":
        each = [work(c) for c in _request_cases(case)]
        return {k: sum(w[k] for w in each) for k in ("bytes", "flops")}
    points = case["rows"] * case["nx"] * case.get("ny", 1)
    cs = 16 if case.get("precision") == "fp64" else 8
    io = 16 if case.get("api") == "host" else cs
    every = case.get("record_every", 0)
    n_rec = case["nz"] // every if every else 0
    stages = STAGES[case["split"]]
    ffts = sum(1 for a, _ in stages if a != 0.0)
    # two bands, a forward and an inverse transform each; the coupling of a
    # cell and the propagator of two modes
    flops = ffts * (20.0 * math.log2(case["nx"] * case.get("ny", 1)) + 12.0) + 32.0 * len(stages)
    flops *= points * case["nz"]
    nbytes = points * 2 * (2 * io + n_rec * cs)
    if case.get("geometry") == "pulse":
        flops += 2 * points * 5.0 * math.log2(case["rows"])
        nbytes += 2 * points * cs * 2
    return {"bytes": nbytes, "flops": flops}


# ---- the same outputs in 64 bits with torch alone -----------------------------


def _bessel(nu, w):
    half = w / 2.0
    term = half ** nu
    total = term
    for m in range(1, 40):
        term = term * (-(half * half)) / (m * (m + nu))
        total += term
    return total


def _reduced_exp(phase):
    return torch.polar(torch.ones_like(phase), torch.remainder(phase, 2.0 * math.pi))


class _Exact:
    """Plain complex128 march of one problem."""

    def __init__(self, case, p):
        self.case, self.p = case, p
        self.dev = "cuda" if torch.cuda.is_available() else "cpu"
        f64 = dict(dtype=torch.float64, device=self.dev)
        nx, ny, rows = p["nx"], p["ny"], p["rows"]
        e = torch.as_tensor(p["energies"], **f64)
        k = 2.0 * math.pi / (HC_EV_ANGSTROM / e * 1e-4)
        s = math.sin(p["theta"]) * p["e_ref"] / e
        c = torch.sqrt((1.0 - s) * (1.0 + s))
        self.k_dz = (k * p["dz"]).tolist()
        self.cos = c.tolist()
        qx = 2.0 * math.pi * torch.fft.fftfreq(nx, d=1.0, **f64)[None] / (k[:, None] * p["dx"])
        qx = qx[:, None, :]
        qy2 = torch.zeros(1, 1, 1, **f64)
        if ny > 1:
            qy = 2.0 * math.pi * torch.fft.fftfreq(ny, d=1.0, **f64)[None] / (k[:, None] * p["dy"])
            qy2 = (qy ** 2)[:, :, None]
        s, c = s[:, None, None], c[:, None, None]
        self.delta, self.root_c = [], c
        for sign in (1.0, -1.0):
            root = torch.sqrt(1.0 - (qx + sign * s) ** 2 - qy2)
            self.delta.append(-(qx * (qx + sign * 2.0 * s) + qy2) / (root + c))
        self.delta = torch.stack(self.delta, 1)          # [B][2][ny][nx]
        self.kd = (k * p["dz"])[:, None, None, None]
        d_um = HC_EV_ANGSTROM / p["e_ref"] * 1e-4 / (2.0 * math.sin(p["theta"]))
        self.h = 2.0 * math.pi / d_um
        self.x = p["x0"] + torch.arange(nx, **f64) * p["dx"]
        self.y = (p["y0"] + torch.arange(ny, **f64) * p["dy"])[:, None] if ny > 1 else torch.zeros(1, 1, **f64)

    def coupling(self, frac):
        """(a, b) of every row for a step of frac dz, [B][1][1]."""
        a, b = [], []
        for kdz, c in zip(self.k_dz, self.cos):
            w = frac * kdz * self.p["chih"] / c
            phi = cmath.exp(1j * frac * kdz * self.p["chi0"] / (2.0 * c))
            a.append(_bessel(0, w) * phi)
            b.append(1j * _bessel(1, w) * phi)
        t = lambda v: torch.tensor(v, dtype=torch.complex128, device=self.dev)[:, None, None]  # noqa: E731
        return t(a), t(b)

    def slices(self, n0, n1):
        """Phasors exp(i h u) of steps [n0, n1), zero outside the crystal: [n][ny][nx]."""
        p = self.p
        z = (torch.arange(n0, n1, dtype=torch.float64, device=self.dev) * p["dz"])[:, None, None]
        x, s = self.x[None, None], p["slab"]
        if s["kind"] == VACUUM:
            inside = torch.zeros_like(z + x, dtype=torch.bool)
        elif s["kind"] == BOX:
            b, y = s["box"], self.y[None]
            inside = ((x >= b[0]) & (x <= b[1]) & (y >= b[2]) & (y <= b[3]) & (z >= b[4]) & (z <= b[5]))
        else:
            n = [v if abs(v) >= 1e-12 else 0.0 for v in (math.cos(s["angle"]), math.sin(s["angle"]))]
            depth = n[0] * (x - s["surf"][0]) + n[1] * (z - s["surf"][1])
            inside = (depth >= 0.0) & (depth <= s["thick"])
            if s["kind"] == SLAB_AND_POLYGON:
                poly, odd = s["polygon"], torch.zeros_like(inside)
                for i in range(len(poly)):
                    (xa, za), (xb, zb) = poly[i - 1], poly[i]
                    cross = (z < za) != (z < zb)
                    odd ^= cross & (x < (xb - xa) * (z - za) / (zb - za) + xa)
                inside = inside & odd
        kind, q = p["strain"]
        if kind == BENT:
            ph = _reduced_exp(self.h * ((x - q[2]) ** 2 + q[1] * (z - q[3]) ** 2) / (2.0 * q[0]))
        elif kind == DISLOCATION:
            xx, zz = x - q[2], z - q[3]
            u = q[0] / (2.0 * math.pi) * (torch.atan2(zz, xx) + xx * zz / (2.0 * (1.0 - q[1]) * (xx ** 2 + zz ** 2)))
            ph = _reduced_exp(self.h * u)
        else:
            ph = torch.ones_like(z + x, dtype=torch.complex128)
        return torch.where(inside, ph, torch.zeros_like(ph)).expand(n1 - n0, max(p["ny"], 1), p["nx"])

    def march(self, psi):
        """(final field, records, powers): psi [B][2][ny][nx] complex128."""
        p, case = self.p, self.case
        every = case.get("record_every", 0)
        area = p["dx"] * p.get("dy", 1.0)
        axes = (-2, -1) if p["ny"] > 1 else (-1,)
        stages = []
        for a, b in STAGES[case.get("split", "first")]:
            prop = torch.exp(1j * a * self.kd * self.delta) if a != 0.0 else None
            stages.append((prop, *self.coupling(b)))
        vacuum = p["slab"]["kind"] == VACUUM
        recs, pows = [], []
        chunk = max(1, min(256, (1 << 24) // (p["nx"] * p["ny"])))

        def phase(n):   # the phase that every mode has in common, exp(i n dz^ cos(alpha))
            g = [cmath.exp(1j * math.fmod(n * math.fmod(kd * c, 2.0 * math.pi), 2.0 * math.pi))
                 for kd, c in zip(self.k_dz, self.cos)]
            return torch.tensor(g, dtype=torch.complex128, device=self.dev)[:, None, None, None]

        for n in range(p["nz"]):
            if n % chunk == 0:
                sl = self.slices(n, min(p["nz"], n + chunk))
                inside = sl != 0
            e, m = sl[n % chunk], inside[n % chunk]
            for prop, a, b in stages:
                if prop is not None:
                    f = torch.fft.fftn(psi, dim=axes)
                    psi = torch.fft.ifftn(f.mul_(prop), dim=axes)
                if not vacuum:
                    be, bc, am = b * e, b * e.conj(), torch.where(m, a, torch.ones_like(a))
                    u, v = psi[:, 0], psi[:, 1]
                    psi = torch.stack([am * u + be * v, am * v + bc * u], 1)
            if every and (n + 1) % every == 0:
                recs.append(psi * phase(n + 1))
                pows.append(psi.abs().square().sum((-2, -1)) * area)
        pows.append(psi.abs().square().sum((-2, -1)) * area)
        psi = psi * phase(p["nz"])
        return psi, torch.stack(recs, 1) if recs else None, torch.stack(pows, 1)


def _exact_march(case, seed):
    p = _setup_cube(case, seed) if case["kind"] == "cube" else _setup(case, seed)
    m = _Exact(case, p)
    psi = torch.from_numpy(p["psi"])
    if case.get("precision") != "fp64":
        psi = psi.to(torch.complex64)      # what a single-precision march is given
    psi = psi.to(device=m.dev, dtype=torch.complex128)
    if p["ny"] == 1:
        psi = psi[:, :, None, :]
    out, recs, pows = m.march(psi)
    if p["ny"] == 1:
        out = out[:, :, 0]
        recs = None if recs is None else recs[:, :, :, 0]
    return out, recs, pows


def exact(case, seed):
    if case["kind"] == "serve":
        if sum(c["nz"] for c in _request_cases(case)) > 120_000:
            return None
        return [_exact_march(c, seed * 1000 + i)[0].cpu() for i, c in enumerate(_request_cases(case))]
    out, recs, pows = _exact_march(case, seed)
    if case.get("api") == "host":
        if recs is None:
            recs = torch.zeros((out.shape[0], 0) + tuple(out.shape[1:]), dtype=torch.complex128)
        return [out, recs, pows]
    outs = [out] if recs is None else [out, recs]
    if case.get("geometry") == "rocking":
        outs.append(pows)
    if case.get("geometry") == "pulse":
        # the superposition of the monochromatic solutions exp(-i omega_j t)
        outs.append(torch.fft.fft(out, dim=0).permute(1, 2, 0).contiguous())
    return outs
