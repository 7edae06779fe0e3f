"""The measured workloads of the screened-WKB library: what its users run, through its public entry
points (``paper_2301_03814_gb300.swkb``), from one pruned DFT to a paper-scale duct.

A case is a dict of plain values; its "kind" says which entry point it goes through:

  modes   swkb_modes_noalloc: the pruned DFT of one device field, nothing allocated
  field   Plan.propagate_device: a field carried over a number of screens
  planes  Plan.propagate_planes_device: the fields on planes between the screens
  batch   Batch.run_device: many uneven propagations in one persistent launch
  serve   Server.submit / Server.poll: uneven requests with host buffers
  hill    swkb_hill_propagate_device: the separation-of-variables field

Fields of mixed plans are FP32 numbers handed over as complex128; they are returned as complex64, which
holds each of them exactly.  FP64 plans' fields are returned as they come.
"""
from __future__ import annotations

import decimal
import functools
import math

import numpy as np
import torch

from paper_2301_03814_gb300 import swkb
from paper_2301_03814_gb300 import workloads as w

BCS = {"periodic": w.BC_PERIODIC, "neumann": w.BC_NEUMANN, "dirichlet": w.BC_DIRICHLET}


def listed():
    return [
        # Step (a) alone, for a host framework that owns all device memory: the smallest call there is.
        {"name": "modes-4096", "kind": "modes", "n_fft": 4096, "n_max": 244},
        # The unit-wavelength check case a new user runs first: FP64, ten short screens, latency-bound.
        {"name": "unit-512-fp64", "kind": "field", "medium": "unit", "precision": "fp64", "n_z": 512,
         "screens": 10, "q0": 0},
        # The 40 km lens like the paper's first example: x-invariant, so its rays are marched once per call
        # (reuse_rays); the rest is DFT, sum and launches.
        {"name": "lens-4096-reuse", "kind": "field", "medium": "lens", "precision": "mixed", "n_z": 4096,
         "screens": 40, "q0": 0, "reuse": True},
        # A small surface duct (50 m high): the size of an interactive run.
        {"name": "duct-4096-mixed", "kind": "field", "medium": "duct", "bc": "neumann", "precision": "mixed",
         "n_z": 4096, "screens": 12, "q0": 0},
        # The surface duct of the headline benchmark: N_z = 16384, 977 modes, Neumann ground, absorber.
        {"name": "duct-16384-mixed", "kind": "field", "medium": "duct", "bc": "neumann", "precision": "mixed",
         "n_z": 16384, "screens": 20, "q0": 0},
        # The same in FP64, the accuracy reference of a mixed production run.
        {"name": "duct-16384-fp64", "kind": "field", "medium": "duct", "bc": "neumann", "precision": "fp64",
         "n_z": 16384, "screens": 2, "q0": 0},
        # Paper scale: N_z = 131072, the duct varies over the range (several table columns), resumed half-way.
        {"name": "duct-131072-range", "kind": "field", "medium": "range", "precision": "mixed",
         "n_z": 131072, "screens": 6, "q0": 100},
        # Pictures of the field between the screens: four planes per screen, Dirichlet ground.
        {"name": "planes-8192-mixed", "kind": "planes", "medium": "duct", "bc": "dirichlet",
         "precision": "mixed", "n_z": 8192, "screens": 3, "q0": 0, "planes": 4},
        # Overlapping Fourier continuation on an open interval of 43 690 wavelengths, 188 patches.
        {"name": "open-131072-mixed", "kind": "field", "medium": "open", "precision": "mixed",
         "n_z": 131072, "patch": 920, "overlap": 224, "stride": 8, "screens": 4, "q0": 0},
        # The uneven batch: instances of mixed frequency, N_z, range and duct in one launch.
        {"name": "batch-12-mixed", "kind": "batch", "precision": "mixed", "mix": 4, "count": 12,
         "n_z_lo": 4096, "n_z_hi": 32768, "screens_lo": 3, "screens_hi": 8},
        # A burst of served requests of mixed sizes, host field in, host field out.
        {"name": "serve-8-mixed", "kind": "serve", "precision": "mixed", "mix": 5, "count": 8,
         "n_z_lo": 4096, "n_z_hi": 16384, "screens_lo": 8, "screens_hi": 20},
        # The exact one-way field of the surface duct at 1 and 2 km, 641 modes (separation of variables).
        {"name": "hill-640", "kind": "hill", "bc": "neumann", "n_z": 16384, "K": 640, "n_q": 32768,
         "batch": 1, "ranges": 2, "x_max": 2000.0},
    ]


def _log2(rng, lo, hi):
    return 1 << int(math.floor(rng.uniform(math.log2(lo), math.log2(hi) + 0.9999)))


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["modes", "unit", "lens", "duct", "duct", "duct", "range", "planes", "open", "open",
                       "batch", "serve", "hill"])
    if kind == "modes":
        n = _log2(rng, 256, 65536)
        return {"kind": "modes", "n_fft": n, "n_max": _log(rng, max(1, n // 64), n // 4 - 1)}
    if kind == "unit":
        return {"kind": "field", "medium": "unit", "precision": rng.choice(["fp64", "mixed"]),
                "n_z": rng.choice([256, 512, 1024]), "screens": rng.randint(1, 10), "q0": rng.randint(0, 9)}
    if kind == "lens":
        return {"kind": "field", "medium": "lens", "precision": rng.choice(["fp64", "mixed", "mixed"]),
                "n_z": rng.choice([2048, 4096, 8192]), "screens": rng.randint(2, 10), "q0": 0,
                "reuse": rng.random() < 0.5}
    if kind == "duct":
        precision = rng.choice(["fp64", "mixed", "mixed"])
        n = _log2(rng, 2048, 8192 if precision == "fp64" else 32768)
        return {"kind": "field", "medium": "duct", "bc": rng.choice(["neumann", "neumann", "dirichlet"]),
                "precision": precision, "n_z": n, "screens": rng.randint(1, max(1, (1 << 15) // n)) if
                precision == "fp64" else rng.randint(1, 12), "q0": rng.randint(0, 50),
                "stride": rng.choice([8, 16, 32]), "steps": rng.choice([12, 16])}
    if kind == "range":
        return {"kind": "field", "medium": "range", "precision": "mixed", "n_z": _log2(rng, 16384, 131072),
                "screens": rng.randint(1, 5), "q0": rng.randint(0, 150)}
    if kind == "planes":
        return {"kind": "planes", "medium": "duct", "bc": rng.choice(["neumann", "dirichlet"]),
                "precision": "mixed", "n_z": _log2(rng, 2048, 8192), "screens": rng.randint(1, 3), "q0": 0,
                "planes": rng.choice([2, 4, 8])}
    if kind == "open":
        precision = rng.choice(["fp64", "mixed", "mixed"])
        overlap, patches = rng.randint(160, 260), _log(rng, 2, 8 if precision == "fp64" else 120)
        patch = rng.randint(2 * overlap + 60, 920)
        while -(patch + (patches - 1) * (patch - overlap)) % 64 > 12:   # the lens's table reaches that far
            overlap, patch = overlap + 1, patch + rng.choice([2, 3])
        return {"kind": "field", "medium": "open", "precision": precision,
                "n_z": patch + (patches - 1) * (patch - overlap), "patch": patch, "overlap": overlap,
                "stride": rng.choice([2, 4, 8]) if patches < 20 else 8, "screens": rng.randint(1, 3), "q0": 0}
    if kind == "batch":
        return {"kind": "batch", "precision": "mixed",
                "mix": rng.randint(10, 10000), "count": rng.randint(3, 8), "n_z_lo": 4096, "n_z_hi": 8192,
                "screens_lo": 1, "screens_hi": 4}
    if kind == "serve":
        return {"kind": "serve", "precision": "mixed", "mix": rng.randint(10, 10000),
                "count": rng.randint(2, 6), "n_z_lo": 4096, "n_z_hi": 8192, "screens_lo": 4,
                "screens_hi": 12}
    K = rng.randint(40, 420)
    return {"kind": "hill", "bc": rng.choice(["neumann", "dirichlet", "periodic"]), "n_z": rng.choice([2048, 4096, 8192]),
            "K": K, "n_q": 4096, "batch": rng.choice([1, 1, 2, 3]), "ranges": rng.randint(1, 3),
            "x_max": float(rng.randint(100, 1000))}


# --------------------------------------------------------------------------------------------------
# inputs
# --------------------------------------------------------------------------------------------------

def _problem(case, seed):
    """The workloads.Problem of a "field" or "planes" case; the seed moves the source and, for ducts, the
    duct's top and gradient."""
    rng = np.random.default_rng(1000 + seed)
    n_z, med = case["n_z"], case["medium"]
    if med == "unit":
        pb = w.config_unit_periodic()
        z = 64.0 / n_z * np.arange(n_z)
        u0 = w.gaussian_beam(z, pb.k, rng.uniform(26.0, 38.0), rng.uniform(3.5, 5.0),
                             math.radians(rng.uniform(-3.0, 3.0)))
        return pb.with_(n_z=n_z, u0=u0)
    if med == "lens":
        pb = w.config_gaussian_lens_40km()
        z = pb.z_a + (pb.z_b - pb.z_a) / n_z * np.arange(n_z)
        return pb.with_(n_z=n_z, u0=w.gaussian_beam(z, pb.k, rng.uniform(-20.0, 20.0), rng.uniform(40.0, 70.0), 0.0))
    if med == "duct":
        height = n_z * 200.0 / 16384
        low = height < 150.0
        kw = dict(height=height, n_z=n_z, z_s=float(rng.uniform(4.0, 6.0) if low else rng.uniform(8.0, 15.0)),
                  z_t_range=(10.0, 20.0) if low else (20.0, 60.0), bc=BCS[case["bc"]],
                  ray_stride=case.get("stride", 16), rk4_steps=case.get("steps", 16))
        return w.config_surface_duct(seed=int(seed), **kw)
    if med == "range":
        return w.config_range_dependent_duct(seed=int(seed), height=n_z * 500.0 / 131072, n_z=n_z,
                                             range_m=10_000.0, n_screens=200,
                                             z_s=float(rng.uniform(15.0, 30.0)))
    return w.config_open_lens(n_z=n_z, fc_patch=case["patch"], fc_overlap=case["overlap"], seed=int(seed),
                              n_beams=max(1, min(8, n_z // 512)), ray_stride=case["stride"])


def _problems(case, seed):
    """The uneven requests of a "batch" or "serve" case: sizes and media from its mix, sources from the seed."""
    shape = np.random.default_rng(case["mix"])
    rng = np.random.default_rng(2000 + seed)
    out = []
    for _ in range(case["count"]):
        pb = w.random_request(shape, n_z_range=(case["n_z_lo"], case["n_z_hi"]), range_km=(5.0, 5.0))
        n = int(shape.integers(case["screens_lo"], case["screens_hi"] + 1))
        u0 = w.antenna_beam(pb.z_phys, pb.k, float(rng.uniform(5.0, 30.0)),
                            math.radians(pb.meta["beamwidth_deg"]), pb.bc)
        out.append(pb.with_(n_screens=n, u0=u0))
    return out


def _hill_inputs(case, seed):
    rng = np.random.default_rng(3000 + seed)
    bc, n_z, n_q = BCS[case["bc"]], case["n_z"], case["n_q"]
    lam = 0.05
    k = 2.0 * math.pi / lam
    if case["bc"] == "periodic":
        z_a, z_b, z_c, half = -200.0, 200.0, 0.0, 200.0
    else:
        z_a, z_b, z_c, half = 0.0, n_z * 200.0 / 16384, 0.0, n_z * 200.0 / 16384
    s = half * np.arange(n_q + 1) / n_q
    z = z_a + (z_b - z_a) / n_z * np.arange(n_z)
    eps, u0 = [], []
    for _ in range(case["batch"]):
        if case["bc"] == "periodic":
            eps.append(w.f_gaussian(1e-4, float(rng.uniform(5e-4, 2e-3)))(s)[0])
            u0.append(w.gaussian_beam(z, k, 0.0, float(rng.uniform(8.0, 12.0)), math.radians(0.2)))
        else:
            top = (10.0, 20.0) if half < 150.0 else (20.0, 60.0)
            eps.append(w.f_trilinear_duct(float(rng.uniform(*top)), float(rng.uniform(-0.2, -0.05)))(s)[0])
            u0.append(w.antenna_beam(z, k, float(rng.uniform(4.0, 10.0)), math.radians(1.0), bc))
    xs = case["x_max"] * np.arange(1, case["ranges"] + 1) / case["ranges"]
    return dict(bc=bc, z_a=z_a, z_b=z_b, z_c=z_c, k=np.full(case["batch"], k), eps=np.array(eps),
                u0=np.array(u0, dtype=np.complex128), xs=xs)


def _modes_input(case, seed):
    """A sum of Gaussian beams of mixed widths and angles on the period, as a screen holds it."""
    rng = np.random.default_rng(4000 + seed)
    n = case["n_fft"]
    m = np.arange(n)
    u = np.zeros(n, dtype=np.complex128)
    for _ in range(6):
        c, width = rng.uniform(0.1, 0.9) * n, rng.uniform(0.005, 0.05) * n + 2.0
        f = rng.uniform(-0.5, 0.5) * case["n_max"] / n
        u += rng.uniform(0.3, 1.0) * np.exp(-((m - c) / width) ** 2 + 2j * math.pi * f * (m - c))
    return u


PRECISION = {"fp64": swkb.SWKB_FP64, "mixed": swkb.SWKB_MIXED}


def prepare(case, seed):
    kind = case["kind"]
    state = {"kind": kind, "case": case, "mixed": case.get("precision") == "mixed"}
    if kind == "modes":
        state["u0"] = torch.from_numpy(_modes_input(case, seed)).cuda()
        state["out"] = torch.empty(2 * case["n_max"] + 1, dtype=torch.complex128, device="cuda")
        return state
    if kind == "hill":
        h = _hill_inputs(case, seed)
        state["desc"] = swkb.hill_desc(h["bc"], h["z_a"], h["z_b"], case["n_z"], case["K"], case["n_q"], h["z_c"])
        state["k"], state["xs"] = h["k"], h["xs"]
        state["eps"], state["u0"] = torch.from_numpy(h["eps"]).cuda(), torch.from_numpy(h["u0"]).cuda()
        state["out"] = torch.empty(case["batch"], case["ranges"], case["n_z"], dtype=torch.complex128, device="cuda")
        return state
    if kind in ("batch", "serve"):
        pbs = _problems(case, seed)
        state["problems"] = pbs
        if kind == "serve":
            state["server"] = swkb.Server(64 << 30, 16)
            return state
        state["batch"] = swkb.Batch(pbs, PRECISION[case["precision"]])
        state["u0"] = torch.from_numpy(np.concatenate([pb.u0 for pb in pbs])).cuda()
        state["out"] = torch.empty_like(state["u0"])
        return state
    pb = _problem(case, seed)
    state["plan"] = swkb.Plan(pb, PRECISION[case["precision"]], reuse_rays=bool(case.get("reuse", False)),
                              planes=case.get("planes", 0))
    rows = case["screens"] * case["planes"] if kind == "planes" else 1
    state["u0"] = torch.from_numpy(np.ascontiguousarray(pb.u0, dtype=np.complex128)).cuda()
    state["out"] = torch.empty(rows, pb.n_z, dtype=torch.complex128, device="cuda")
    return state


def run(state):
    kind, case = state["kind"], state["case"]
    if kind == "serve":
        server, pbs = state["server"], state["problems"]
        tickets = [server.submit(pb, PRECISION[case["precision"]])[1] for pb in pbs]
        got = [server.poll(t)[1] for t in tickets]
        return [g.astype(np.complex64) if state["mixed"] else g for g in got]
    u0, out = state["u0"], state["out"]
    if kind == "modes":
        swkb.check(swkb.swkb_modes_noalloc(u0.data_ptr(), case["n_fft"], case["n_max"], out.data_ptr(),
                                           torch.cuda.current_stream().cuda_stream))
    elif kind == "hill":
        swkb.swkb_hill_propagate_device(state["desc"], state["k"], state["eps"].data_ptr(), u0.data_ptr(),
                                        state["xs"], out.data_ptr())
    elif kind == "batch":
        state["batch"].run_device(u0.data_ptr(), out.data_ptr())
    elif kind == "planes":
        state["plan"].propagate_planes_device(case["planes"], u0.data_ptr(), out.data_ptr(), q0=case["q0"],
                                              n_screens=case["screens"])
    else:
        state["plan"].propagate_device(u0.data_ptr(), out.data_ptr(), q0=case["q0"], n_screens=case["screens"])
    return out.to(torch.complex64) if state["mixed"] else out


# --------------------------------------------------------------------------------------------------
# what a pass cannot do without
# --------------------------------------------------------------------------------------------------

def _shape(pb):
    """Modes, marched modes, rays per mode, period points and summed points of a propagation."""
    lam = 2.0 * math.pi / pb.k
    H = pb.z_b - pb.z_a
    if pb.bc == w.BC_OPEN:
        points, period, N = pb.fc_patch + 25, (pb.fc_patch + 25) * H / pb.n_z, -(-pb.n_z // 64) * 64
    else:
        mirrored = pb.bc != w.BC_PERIODIC
        N = points = pb.n_z * (2 if mirrored else 1)
        period = H * (2 if mirrored else 1)
    n_max = pb.n_max if pb.n_max > 0 else int(math.floor(math.sin(pb.theta_max) * period / lam * (1.0 + 1e-12)))
    n_max = min(n_max, points // 2 - 1)
    kmax = n_max * lam / period
    G = int(math.ceil(pb.dx * kmax / math.sqrt(1.0 - kmax * kmax) / (pb.ray_stride * H / pb.n_z) - 1e-9)) + 3
    return dict(n_max=n_max, M=2 * n_max + 1, rays=-(-N // pb.ray_stride) + 2 * G, N=N, points=points, period=period,
                G=G, marched=n_max + 1 if pb.bc in (w.BC_NEUMANN, w.BC_DIRICHLET) else 2 * n_max + 1)


def _field_work(pb, screens, planes=1, marches=None):
    """Per screen: the DFT (5 N log2 N), 77 flops per RK4 stage and ray, 32 per mode and grid point; the
    input and output fields and the medium table once."""
    g = _shape(pb)
    patches = (pb.n_z - pb.fc_patch) // (pb.fc_patch - pb.fc_overlap) + 1 if pb.bc == w.BC_OPEN else 1
    dft = 5.0 * patches * g["points"] * math.log2(g["points"])
    march = 4.0 * pb.rk4_steps * 77.0 * g["marched"] * g["rays"]
    total = 32.0 * g["M"] * pb.n_z * planes
    return {"bytes": 16.0 * pb.n_z * (1 + (screens * planes if planes > 1 else 1)) + 24.0 * pb.profile.eps.size,
            "flops": screens * (dft + total) + (screens if marches is None else marches) * march}


def work(case):
    kind = case["kind"]
    if kind == "modes":
        n = case["n_fft"]
        return {"bytes": 16.0 * (n + 2 * case["n_max"] + 1), "flops": 5.0 * n * math.log2(n)}
    if kind == "hill":
        n, b = case["K"] + 1, case["batch"] * (2 if case["bc"] == "periodic" else 1)
        # symmetric eigen-decomposition with vectors (9 n^3), projection and synthesis
        return {"bytes": 8.0 * case["batch"] * (case["n_q"] + 1 + 2 * case["n_z"] * (1 + case["ranges"])),
                "flops": b * (9.0 * n ** 3 + 4.0 * n * case["n_z"] * (1 + case["ranges"]))}
    if kind in ("batch", "serve"):
        each = [_field_work(pb, pb.n_screens) for pb in _problems(case, 0)]
        return {k: float(sum(e[k] for e in each)) for k in ("bytes", "flops")}
    return _field_work(_problem(case, 0), case["screens"], case.get("planes", 1), 1 if case.get("reuse") else None)


# --------------------------------------------------------------------------------------------------
# the same values from plain torch in 64 bits
# --------------------------------------------------------------------------------------------------

def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


class _Table:
    """eps - ref and its z-derivatives: quintic Hermite in z, linear in x, even about a ground."""

    def __init__(self, pb):
        p, dev = pb.profile, _device()
        self.z0, self.h, self.ground = p.z0, p.dz, pb.z_a if pb.bc in (w.BC_NEUMANN, w.BC_DIRICHLET) else None
        self.x = np.asarray(p.x_cols, dtype=np.float64)
        self.ref = float(p.eps[0, p.eps.shape[1] // 2])
        f = torch.from_numpy(np.ascontiguousarray(p.eps, dtype=np.float64)).to(dev) - self.ref
        d = torch.from_numpy(np.ascontiguousarray(p.eps_z, dtype=np.float64)).to(dev) * self.h
        s = torch.from_numpy(np.ascontiguousarray(p.eps_zz, dtype=np.float64)).to(dev) * (self.h * self.h)
        f0, f1, d0, d1, s0, s1 = f[:, :-1], f[:, 1:], d[:, :-1], d[:, 1:], s[:, :-1], s[:, 1:]
        jump = f1 - f0
        # the quintic in t in [0, 1] that takes value, slope and curvature at both ends
        self.c = torch.stack([f0, d0, 0.5 * s0,
                              10.0 * jump - 6.0 * d0 - 4.0 * d1 - 1.5 * s0 + 0.5 * s1,
                              -15.0 * jump + 8.0 * d0 + 7.0 * d1 + 1.5 * s0 - s1,
                              6.0 * jump - 3.0 * (d0 + d1) - 0.5 * s0 + 0.5 * s1], dim=-1)

    def weights(self, x, right):
        if len(self.x) == 1:
            return [(0, 1.0)]
        c = int(np.sum(self.x <= x if right else self.x < x)) - 1
        c = min(max(c, 0), len(self.x) - 2)
        span = self.x[c + 1] - self.x[c]
        th = 0.0 if span <= 0 else min(max((x - self.x[c]) / span, 0.0), 1.0)
        return [(i, v) for i, v in ((c, 1.0 - th), (c + 1, th)) if v > 0.0]

    def __call__(self, x, right, z):
        sign = 1.0
        if self.ground is not None:
            sign = torch.where(z < self.ground, -1.0, 1.0)
            z = self.ground + (z - self.ground).abs()
        u = (z - self.z0) / self.h
        i = u.floor().clamp(0, self.c.shape[1] - 1)
        t = u - i
        i = i.long()
        e = ez = ezz = 0.0
        for col, v in self.weights(x, right):
            a = self.c[col][i]
            a0, a1, a2, a3, a4, a5 = a.unbind(-1)
            e = e + v * (a0 + t * (a1 + t * (a2 + t * (a3 + t * (a4 + t * a5)))))
            ez = ez + v * (a1 + t * (2 * a2 + t * (3 * a3 + t * (4 * a4 + t * 5 * a5))))
            ezz = ezz + v * (2 * a2 + t * (6 * a3 + t * (12 * a4 + t * 20 * a5)))
        return e, sign * ez / self.h, ezz / (self.h * self.h)


def _march(table, pb, q, kappa, s, stops):
    """Landing shift z - s, phase excess r - x P_bar and amplitude of the rays (kappa, s) after each number of
    RK4 steps in stops: the x-form ray and variational equations, in deviations from the straight ray."""
    h = pb.dx / pb.rk4_steps
    x0, x1 = pb.x0 + q * pb.dx, pb.x0 + (q + 1) * pb.dx
    pbar2 = table.ref - kappa * kappa
    pbar = pbar2.sqrt()
    last = 2 * pb.rk4_steps

    def medium(l, dz):
        return table(x1, False, s + dz) if l == last else table(x0 + 0.5 * l * h, True, s + dz)

    def slope(l, y):
        dz, dq, _, Z, W = y
        e, ez, ezz = medium(l, dz)
        D = e - dq * (2.0 * kappa + dq)
        P = (pbar2 + D).sqrt()
        Q = kappa + dq
        Ps = (0.5 * ez * Z - Q * W) / P
        return (Q / P, 0.5 * ez / P, D / (P + pbar) + dq * Q / P, (W - Q * Ps / P) / P,
                (0.5 * ezz * Z - 0.5 * ez * Ps / P) / P)

    shape = torch.broadcast_shapes(kappa.shape, s.shape)
    zero = torch.zeros(shape, dtype=torch.float64, device=s.device)
    y = (zero, zero, zero, zero + 1.0, zero)
    P0 = (pbar2 + medium(0, zero)[0]).sqrt()
    out = []
    for n in range(pb.rk4_steps):
        k1 = slope(2 * n, y)
        k2 = slope(2 * n + 1, tuple(a + 0.5 * h * b for a, b in zip(y, k1)))
        k3 = slope(2 * n + 1, tuple(a + 0.5 * h * b for a, b in zip(y, k2)))
        k4 = slope(2 * n + 2, tuple(a + h * b for a, b in zip(y, k3)))
        y = tuple(a + h / 6.0 * (b1 + 2.0 * b2 + 2.0 * b3 + b4) for a, b1, b2, b3, b4 in zip(y, k1, k2, k3, k4))
        if n + 1 in stops:
            e = medium(2 * (n + 1), y[0])[0]
            P1 = (pbar2 + e - y[1] * (2.0 * kappa + y[1])).sqrt()
            out.append((y[0], y[2], (P0 / (P1 * y[3])).sqrt()))
    return out


def _mode_sum(n, amp, shift, excess, a, k, dz, G, R, period, points, chunk=24):
    """sum_n amp-weighted a_n(m) exp(i (2 pi (n m mod period) / period + k excess_n(m))) at the points: 4-point
    Lagrange in the landings of rays -1 .. +2 around each point.  amp: [M] or, per ray, [M, rays]."""
    dev = shift.device
    out = torch.zeros(len(points), dtype=torch.complex128, device=dev)
    launch = (torch.arange(shift.shape[1], device=dev, dtype=torch.float64) - G) * R
    x = points.double()
    chunk = max(1, int(chunk * 131072 / max(len(points), shift.shape[1])))
    for i in range(0, len(n), chunk):
        land = launch + shift[i:i + chunk] / dz
        rows = land.shape[0]
        j = torch.searchsorted(land, x.expand(rows, -1).contiguous(), right=True) - 1
        X = [land.gather(1, j + o) for o in (-1, 0, 1, 2)]
        wgt = []
        for p in range(4):
            v = torch.ones_like(X[0])
            for l in range(4):
                if l != p:
                    v = v * (x - X[l]) / (X[p] - X[l])
            wgt.append(v)
        r = sum(wgt[p] * excess[i:i + chunk].gather(1, j + p - 1) for p in range(4))
        val = a[i:i + chunk] if amp.dim() == 1 else a[i:i + chunk] * amp[i:i + chunk]
        A = sum(wgt[p] * val.gather(1, j + p - 1) for p in range(4))
        turn = torch.remainder(n[i:i + chunk, None] * points[None, :], period).double() * (2.0 * math.pi / period)
        term = A * torch.polar(torch.ones_like(r), turn + k * r)
        out += (amp[i:i + chunk, None] * term).sum(0) if amp.dim() == 1 else term.sum(0)
    return out


@functools.lru_cache(maxsize=1)
def _continuation(d=5, C=25, harmonics=12, per_step=20):
    """[C, d]: the continuation at x = d .. d + C - 1 of the polynomial through samples at x = 0 .. d - 1, blended
    to zero on [d + C, 2 d + C - 1] by the least-squares trigonometric fit of period 2 (d + C); 110 digits."""
    D = decimal.Decimal
    with decimal.localcontext() as ctx:
        ctx.prec = 110

        def arctan_inverse(v):
            total, term, k = D(0), D(1) / v, 0
            while abs(term) > D(10) ** -112:
                total += term / (2 * k + 1) * (-1 if k % 2 else 1)
                term, k = term / (v * v), k + 1
            return total

        pi = 4 * (4 * arctan_inverse(5) - arctan_inverse(239))
        turn = 2 * (d + C) * per_step            # fitting points per period
        th = 2 * pi / turn
        c1, s1, term, k = D(0), D(0), D(1), 0
        while abs(term) > D(10) ** -112:
            if k % 2 == 0:
                c1 += term * (-1 if k % 4 else 1)
            else:
                s1 += term * (-1 if k % 4 == 3 else 1)
            k += 1
            term = term * th / k
        cs, sn = [D(1)], [D(0)]
        for _ in range(turn - 1):
            cs.append(cs[-1] * c1 - sn[-1] * s1)
            sn.append(sn[-1] * c1 + cs[-2] * s1)

        def row(i):
            out = [D(1)]
            for m in range(1, harmonics + 1):
                out += [cs[m * i % turn], sn[m * i % turn]]
            return out

        near = (d - 1) * per_step + 1
        pts = list(range(near)) + [(d + C) * per_step + i for i in range(near)]
        F = [row(i) for i in pts]
        B = len(F[0])
        rhs = []
        for i in range(near):
            x = D(i) / per_step
            line = []
            for p in range(d):
                v = D(1)
                for l in range(d):
                    if l != p:
                        v = v * (x - l) / (p - l)
                line.append(v)
            rhs.append(line)
        # normal equations, Gauss elimination with pivots
        A = [[sum(f[r] * f[c] for f in F) for c in range(B)] + [sum(F[i][r] * rhs[i][p] for i in range(near)) for p in range(d)]
             for r in range(B)]
        for c in range(B):
            top = max(range(c, B), key=lambda r: abs(A[r][c]))
            A[c], A[top] = A[top], A[c]
            for r in range(c + 1, B):
                f = A[r][c] / A[c][c]
                if f:
                    A[r] = [u - f * v for u, v in zip(A[r], A[c])]
        sol = [[D(0)] * d for _ in range(B)]
        for r in range(B - 1, -1, -1):
            for p in range(d):
                sol[r][p] = (A[r][B + p] - sum(A[r][c] * sol[c][p] for c in range(r + 1, B))) / A[r][r]
        grid = [row((d + i) * per_step) for i in range(C)]
        return np.array([[float(sum(g[b] * sol[b][p] for b in range(B))) for p in range(d)] for g in grid])


def _smooth(t):
    t = np.clip(t, 0.0, 1.0)
    with np.errstate(divide="ignore", over="ignore"):
        a, b = np.exp(-1.0 / t), np.exp(-1.0 / (1.0 - t))
    return a / (a + b)


def _reference(pb, q0, screens, planes=1):
    """The fields after each plane of the screens (planes = 1: only the last screen's field)."""
    dev = _device()
    g = _shape(pb)
    table = _Table(pb)
    dz = (pb.z_b - pb.z_a) / pb.n_z
    sign = {w.BC_NEUMANN: 1.0, w.BC_DIRICHLET: -1.0}.get(pb.bc, 0.0)
    z_lo = 2 * pb.z_a - pb.z_b if sign else pb.z_a
    n = torch.arange(-g["n_max"], g["n_max"] + 1, device=dev)
    kappa = 2.0 * math.pi * n.double() / (pb.k * g["period"])
    pbar = (table.ref - kappa * kappa).sqrt()
    s = z_lo + (torch.arange(g["rays"], device=dev, dtype=torch.float64) - g["G"]) * pb.ray_stride * dz
    stops = [pb.rk4_steps * (j + 1) // planes for j in range(planes)]
    points = torch.arange(pb.n_z, device=dev) + (pb.n_z if sign else 0)
    window = None
    if pb.absorber_frac > 0:
        H, f = pb.z_b - pb.z_a, pb.absorber_frac
        d = pb.z_phys - pb.z_a
        wd = np.where(d > (1 - f) * H, np.cos(0.5 * math.pi * (d - (1 - f) * H) / (f * H)) ** 2, 1.0)
        window = torch.from_numpy(wd).to(dev)
    u = torch.from_numpy(np.ascontiguousarray(pb.u0, dtype=np.complex128)).to(dev)
    top = None       # the field at the period's first point (2 z_a - z_b), which has no physical partner
    if pb.bc == w.BC_OPEN:
        cont = torch.from_numpy(_continuation()).to(dev).to(torch.complex128)
        stride, Np = pb.fc_patch - pb.fc_overlap, g["points"]
        P = (pb.n_z - pb.fc_patch) // stride + 1
        start = np.arange(P) * stride
        at = (np.arange(g["rays"]) - g["G"]) * float(pb.ray_stride)
        ramp = pb.fc_overlap - 1
        S = _smooth((at[:, None] - start) / ramp) * (1.0 - _smooth((at[:, None] - (start + pb.fc_patch - 1 - ramp)) / ramp))
        S = torch.from_numpy(S).to(dev).to(torch.complex128)
        start = torch.from_numpy(start).to(dev)
    marched, rays = None, None
    rows = []
    per = max(1, int(4e7 / g["rays"]))           # modes marched at a time
    for q in range(q0, q0 + screens):
        if pb.bc == w.BC_OPEN:
            f = u.unfold(0, pb.fc_patch, stride)
            ext = f[:, -5:] @ cont.T + (f[:, :5].flip(1) @ cont.T).flip(1)
            c = torch.fft.fft(torch.cat([f, ext], dim=1))[:, torch.remainder(n, Np)] / Np
            c = c * torch.polar(torch.ones_like(c.real), -2.0 * math.pi / Np * torch.remainder(n[None, :] * start[:, None], Np).double())
            amp = (S @ c).T.contiguous()
        else:
            full = u
            if sign:
                first = torch.zeros(1, dtype=u.dtype, device=dev) if top is None else top * (1.0 + sign) / 2.0
                u = torch.cat([u[:1] * (1.0 + sign) / 2.0, u[1:]]) if top is not None else u
                full = torch.cat([first, sign * u[1:].flip(0), u])
            amp = torch.fft.fft(full)[torch.remainder(n, g["N"])] / g["N"]
        key = tuple(tuple(table.weights(pb.x0 + q * pb.dx + 0.5 * l * pb.dx / pb.rk4_steps, True)) for l in range(2 * pb.rk4_steps))
        if key != marched or len(table.x) > 1:
            rays = None
            parts = [_march(table, pb, q, kappa[i:i + per, None], s[None, :], stops) for i in range(0, len(n), per)]
            rays = [tuple(torch.cat([p[j][v] for p in parts]) for v in range(3)) for j in range(planes)]
            del parts
            marched = key
        for j in range(planes):
            shift, excess, a = rays[j]
            base = torch.remainder(pb.k * pb.dx * (j + 1) / planes * pbar, 2.0 * math.pi)
            carry = torch.polar(torch.ones_like(base), base)
            weighted = amp * (carry[:, None] if amp.dim() == 2 else carry)
            pts = torch.cat([points, torch.zeros(1, dtype=points.dtype, device=dev)]) if sign else points
            v = _mode_sum(n, weighted, shift, excess, a, pb.k, dz, g["G"], pb.ray_stride, g["points"], pts)
            top_v = v[-1:] if sign else None
            v = v[:pb.n_z]
            if j == planes - 1 and window is not None:
                v = v * window
                top_v = top_v * 0.0 if sign else None      # the absorber vanishes at the full height
            shown = torch.cat([v[:1] * (1.0 + sign) / 2.0, v[1:]]) if sign else v
            if planes > 1 or q == q0 + screens - 1:
                rows.append(shown)
        u, top = v, top_v
    return torch.stack(rows)


def _hill_reference(case, seed):
    h, dev = _hill_inputs(case, seed), _device()
    n_z, K, n_q = case["n_z"], case["K"], case["n_q"]
    mirrored = case["bc"] != "periodic"
    N = 2 * n_z if mirrored else n_z
    L = (h["z_b"] - h["z_a"]) * (2 if mirrored else 1)
    centre = n_z if mirrored else int(round((h["z_c"] - h["z_a"]) / (L / N)))
    parities = {"neumann": (0,), "dirichlet": (1,), "periodic": (0, 1)}[case["bc"]]
    out = torch.zeros(case["batch"], case["ranges"], n_z, dtype=torch.complex128, device=dev)
    xs = torch.from_numpy(h["xs"]).to(dev)
    at = torch.arange(N, device=dev) - centre
    for b in range(case["batch"]):
        e, k = torch.from_numpy(h["eps"][b]).to(dev), float(h["k"][b])
        mean = torch.fft.rfft(torch.cat([e, e[1:-1].flip(0)])).real[:2 * K + 1] / (2 * n_q)
        u = torch.from_numpy(h["u0"][b]).to(dev)
        if mirrored:
            sg = 1.0 if case["bc"] == "neumann" else -1.0
            u = torch.cat([torch.zeros(1, dtype=u.dtype, device=dev), sg * u[1:].flip(0), u])
        for odd in parities:
            n = torch.arange(odd, K + 1, device=dev)
            norm = torch.where(n == 0, 0.0, 1.0).double() * (math.sqrt(2.0) - 1.0) + 1.0
            A = (mean[(n[:, None] - n[None, :]).abs()] + (-1.0 if odd else 1.0) * mean[n[:, None] + n[None, :]])
            A = 0.5 * k * k * norm[:, None] * norm[None, :] * A - torch.diag((2.0 * math.pi / L * n.double()) ** 2)
            lam, V = torch.linalg.eigh(A.cpu())
            lam, V = lam.to(dev), V.to(dev).to(torch.complex128)
            angle = torch.remainder(n[:, None] * at[None, :], N).double() * (2.0 * math.pi / N)
            E = (norm[:, None] * (angle.sin() if odd else angle.cos())).to(torch.complex128)
            a = V.T @ (E @ u / N)
            alpha = torch.sqrt(lam.to(torch.complex128))
            g = (a[None, :] * torch.exp(1j * alpha[None, :] * xs[:, None])) @ V.T
            field = g @ E
            out[b] += field[:, centre:centre + n_z] if mirrored else field
    return out


def exact(case, seed):
    kind = case["kind"]
    if kind == "modes":
        n, n_max = case["n_fft"], case["n_max"]
        c = np.fft.fft(_modes_input(case, seed)) / n
        return torch.from_numpy(np.concatenate([c[n - n_max:], c[:n_max + 1]]))
    if kind == "hill":
        return _hill_reference(case, seed)
    if kind in ("batch", "serve"):
        fields = [_reference(pb, 0, pb.n_screens)[0] for pb in _problems(case, seed)]
        return torch.cat(fields) if kind == "batch" else [f.cpu().numpy() for f in fields]
    return _reference(_problem(case, seed), case["q0"], case["screens"], case.get("planes", 1))
