"""Timed cases of the fast-electron step: what a program that uses this library has it do.

A pass restores the electrons of a run from page-locked host arrays, advances
a number of steps and reads back what such a program dumps (fields,
temperature, energy budget, and the electrons or the photon spectrum where it
wants them).  Restoring the electrons keeps every pass at the same point of
the run.  Results of an FP32 run are kept in single precision.

The electrons stand in for a run in flight: injected through the laser disc
into the cone, part of them scattered, refluxing between the faces, sorted by
cell as a run leaves them.  `exact` is the same method written in plain
64-bit torch.
"""
from __future__ import annotations

import ctypes
import math

import numpy as np
import torch

from paper_2107_01723_gb300 import hpic
from paper_2107_01723_gb300 import workloads as W

QE, ME, CL, EPS0 = 1.602176634e-19, 9.1093837015e-31, 299792458.0, 8.8541878128e-12
HPL, KB, AMU, A_BOHR = 6.62607015e-34, 1.380649e-23, 1.66053906660e-27, 5.29177210903e-11
HBAR, MU0, MC2 = HPL / (2 * math.pi), 1 / (EPS0 * CL * CL), ME * CL * CL
KEYS = ("x", "y", "z", "ux", "uy", "uz", "tau")
BUDGET = hpic._TALLY_NAMES
PLAIN, SCREENED, EMISSION = 63, 63 | 128 | 256, 1 | 2 | 4 | 64  # physics switches


def listed() -> list:
    def step(name, n, electrons, steps, precision="fp32", sort=3, material="Au", intensity=1e20,
             inject="none", physics="plain", electrons_out=False, spectrum=False):
        return dict(name=name, kind="step", nx=n[0], ny=n[1], nz=n[2], electrons=electrons, steps=steps,
                    precision=precision, sort=sort, material=material, intensity=intensity, inject=inject,
                    physics=physics, electrons_out=electrons_out, spectrum=spectrum)

    return [
        # a few tiles: the smallest useful run (a quick look, a test): launches count
        step("few_tiles_fp32", (10, 9, 11), 2000, 40, sort=0, electrons_out=True, spectrum=True),
        # 32^3 gold, 1e5 electrons at 1e20 W/cm^2: the ordinary small run, and in the plain FP64 path
        step("small_fp32", (32, 32, 32), 100_000, 30),
        step("small_fp64", (32, 32, 32), 100_000, 10, precision="fp64", sort=0, electrons_out=True, spectrum=True),
        # 64^3 in FP64: a reference run that single precision is checked against
        step("medium_fp64", (64, 64, 64), 1_000_000, 5, precision="fp64", intensity=1e21, spectrum=True),
        # the benchmark: 128^3 gold, 1e7 electrons at 1e21 W/cm^2
        step("headline_fp32", (128, 128, 128), 10_000_000, 30, intensity=1e21),
        # a thick target while its laser is on: a large grid with few electrons yet, more every step
        step("thick_injecting_fp32", (250, 126, 130), 1_000_000, 40, intensity=1e22, inject="flat"),
        # ionised-screening cross section and electron-ion equilibration, ragged sizes
        step("screened_fp32", (45, 61, 52), 300_000, 20, material="Al", intensity=1e21, physics="screened"),
        # CH plastic under the Gaussian envelope: weighted electrons, two elements per cell
        step("plastic_gauss_fp32", (60, 50, 47), 400_000, 10, material="CH", intensity=1e21, inject="gauss"),
        # a parameter scan advanced as one batch, and a small uneven one
        dict(name="scan_fp32", kind="batch", targets=16, cross=64, thin=5, thick=200, electrons=8_000_000, steps=30,
             blocks=2, sort=3, precision="fp32"),
        dict(name="small_scan_fp32", kind="batch", targets=5, cross=12, thin=6, thick=15, electrons=30_000, steps=30,
             blocks=2, sort=3, precision="fp32"),
        # the emission benchmark: unbounded gold, collisions and photons only
        dict(name="emission_fp32", kind="emission", electrons=1 << 23, steps=20, precision="fp32"),
        # the loss-channel heatmap over intensity and Z
        dict(name="heatmap", kind="model", intensities=64, elements=92),
    ]


def draw(rng) -> dict:
    def between(lo, hi):  # spread over the logarithm
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["step", "step", "step", "step64", "batch", "emission", "model"])
    if kind == "step":
        n = [between(6, 160) for _ in range(3)]
        electrons = between(1000, 4_000_000)
        physics = rng.choice(["plain", "plain", "screened"])
        material = rng.choice(["Au", "Cu", "Al"] if physics == "screened" else ["Au", "Cu", "Al", "CH"])
        small = electrons <= 5000
        return dict(kind="step", nx=n[0], ny=n[1], nz=n[2], electrons=electrons, steps=rng.randint(4, 25),
                    precision="fp32", sort=0 if small else rng.choice([2, 3, 5]), material=material,
                    intensity=10 ** rng.uniform(20, 22), inject=rng.choice(["none", "none", "flat", "gauss"]),
                    physics=physics, electrons_out=small, spectrum=False)
    if kind == "step64":
        n = [between(6, 80) for _ in range(3)]
        return dict(kind="step", nx=n[0], ny=n[1], nz=n[2], electrons=between(1000, 600_000), steps=rng.randint(2, 6),
                    precision="fp64", sort=0, material=rng.choice(["Au", "Cu", "Al", "CH"]),
                    intensity=10 ** rng.uniform(20, 22), inject=rng.choice(["none", "flat"]), physics="plain",
                    electrons_out=True, spectrum=True)
    if kind == "batch":
        targets, thin = rng.randint(1, 16), rng.randint(5, 30)
        cross = between(10, 64)
        return dict(kind="batch", targets=targets, cross=cross, thin=thin, thick=thin + between(4, 150),
                    electrons=targets * between(2000, 400_000), steps=rng.randint(5, 25), blocks=rng.randint(1, 5),
                    sort=rng.choice([0, 3, 5]), precision="fp32")
    if kind == "emission":
        precision = rng.choice(["fp32", "fp32", "fp64"])
        return dict(kind="emission", electrons=between(3000, 1 << 23 if precision == "fp32" else 1 << 20),
                    steps=rng.randint(3, 15 if precision == "fp32" else 5), precision=precision)
    return dict(kind="model", intensities=between(1, 64), elements=rng.randint(1, 92))


# ---------------------------------------------------------------- inputs
def target_of(case: dict) -> dict:
    n = (case["nx"], case["ny"], case["nz"])
    if case["material"] == "CH":
        return W.compound([("C", None), ("H", None)], n=n)
    return W.target(n=n, material=case["material"])


def macro_electrons(n: int, intensity: float) -> int:
    """Macro-electrons of the laser: those in flight, or more of them where these would weigh too much each."""
    return max(n, int(2e5 * math.sqrt(intensity / 1e20)))


def laser_of(case: dict, t: dict) -> dict:
    spot = min(5.0, 0.4 * min(case["ny"], case["nz"])) * 1e-6
    if case["inject"] == "gauss":
        return W.laser_gauss(t, I_Wcm2=case["intensity"], per_cell=max(2, min(1226, case["electrons"] // 400)),
                             r_fwhm=1.02 * spot)  # no cell centre on the edge of the spot
    n = macro_electrons(case["electrons"], case["intensity"]) * (1 if case["inject"] == "none" else 5)
    return W.laser(t, I_Wcm2=case["intensity"], n_macro=n, spot_r=spot)


def run_of(case: dict, seed: int, target_index: int = 0) -> dict:
    physics = {"plain": PLAIN, "screened": SCREENED, "emission": EMISSION}[case.get("physics", "plain")]
    return W.run(seed=seed, physics=physics, max_history=400, target_index=target_index)


def first_step(case: dict) -> int:
    return 20 if case.get("inject", "none") != "none" else 300  # inside, or past, the injection window


def mean_energy(intensity: float) -> float:
    return 8.5e-6 * math.sqrt(intensity * 1e4 * 1e-12)  # a0 of Eq. (1): T_hot in m_e c^2


def device() -> torch.device:
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def electrons(n, cells, mean, spot, seed, real) -> dict:
    """Electrons of a run in flight, in cells and m_e c, sorted by cell tiles: `real`-precision values."""
    dev = device()
    g = torch.Generator(device=dev).manual_seed(seed)

    def rand():
        return torch.rand(n, generator=g, device=dev, dtype=torch.float64)

    if spot is None:  # uniform and isotropic
        pos = [c * rand() for c in cells]
        s = torch.full_like(pos[0], 1e9)
    else:
        r, phi = spot * torch.sqrt(rand()), 2 * math.pi * rand()
        pos = [torch.full_like(r, 1e-3), 0.5 * cells[1] + r * torch.cos(phi), 0.5 * cells[2] + r * torch.sin(phi)]
        s = 0.8 * max(min(cells), cells[0]) * rand()
    ct, phi = 1 - (1 - math.cos(math.radians(30))) * rand(), 2 * math.pi * rand()
    iso = rand() < (0.3 if spot is not None else 2.0)
    ct = torch.where(iso, 2 * rand() - 1, ct)
    st = torch.sqrt(1 - ct * ct)
    d = [ct, st * torch.cos(phi), st * torch.sin(phi)]
    if spot is not None:  # fly, scatter a little, reflect at the faces
        pos = [p + s * q for p, q in zip(pos, d)]
        a = 0.1 * torch.sqrt(s / 20)
        d = [q + a * torch.randn(n, generator=g, device=dev, dtype=torch.float64) for q in d]
        for c in range(3):
            turns = torch.floor(pos[c] / cells[c])
            f = pos[c] - turns * cells[c]
            odd = torch.remainder(turns, 2) != 0
            pos[c] = torch.where(odd, cells[c] - f, f)
            d[c] = torch.where(odd, -d[c], d[c])
    norm = torch.sqrt(sum(q * q for q in d))
    eps = 0.04 - mean * torch.log1p(-rand())
    u = torch.sqrt(eps * (eps + 2))
    tau = -torch.log1p(-rand())
    pos = [torch.clamp(p, 1e-3, c - 1e-3) for p, c in zip(pos, cells)]
    cell = [p.long() for p in pos]
    nt = [(c + 3) // 4 for c in cells]
    tile = (cell[2] // 4 * nt[1] + cell[1] // 4) * nt[0] + cell[0] // 4
    order = torch.argsort(tile * 64 + cell[2] % 4 * 16 + cell[1] % 4 * 4 + cell[0] % 4, stable=True)
    values = pos + [u * q / norm for q in d] + [tau]
    out = {k: v[order].to(real).double() for k, v in zip(KEYS, values)}
    out["w"] = (2e6 * (0.5 + rand())).to(real).double()  # used where electrons carry their own weight
    out["id"] = torch.arange(n, device=dev)
    return out


def page_locked(p: dict, dx: float) -> dict:
    out = {}
    for k in (k for k in KEYS + ("id", "w") if k in p):
        v = p[k]
        v = (v * dx if k in "xyz" else v).to(torch.int32 if k == "id" else torch.float64)
        h = torch.empty(v.shape, dtype=v.dtype, pin_memory=torch.cuda.is_available())
        h.copy_(v)
        out[k] = h.numpy().view(np.uint32) if k == "id" else h.numpy()
    return out


def fields(t: dict, seed: int) -> dict:
    """Smooth live fields (SI): E of 1e9 V/m, B of 1000 T, T from 20 to 200 eV (T_i below it), eta(T)."""
    rng = np.random.default_rng(seed)
    n = (t["nz"] + 1, t["ny"] + 1, t["nx"] + 1)

    def wave(shape):
        a = [np.sin(2 * math.pi * (rng.uniform(0.5, 2) * np.arange(m) / m + rng.uniform())) for m in shape]
        return a[0][:, None, None] * a[1][None, :, None] * a[2][None, None, :]

    out = {c: 1e9 * wave(n) for c in ("Ex", "Ey", "Ez")}
    out.update({c: 1000.0 * wave(n) for c in ("Bx", "By", "Bz")})
    c = (t["nz"], t["ny"], t["nx"])
    out["T"] = (110.0 + 90.0 * wave(c)) * W.KELVIN_PER_EV
    out["Ti"] = 0.5 * out["T"] * (1.0 + 0.3 * wave(c))
    out["eta"] = Solid(t).resistivity(torch.from_numpy(out["T"])).numpy()
    return out


def batch_of(case: dict, seed: int):
    cfg = W.config4(n_targets=case["targets"], total_macro=case["electrons"],
                    lo=case["electrons"] // (4 * case["targets"]), hi=4 * case["electrons"] // case["targets"],
                    cross=case["cross"], thickness=(case["thin"], case["thick"]))
    counts = [l["n_macro"] for l in cfg["lasers"]]
    for l, n, I in zip(cfg["lasers"], counts, cfg["I_Wcm2"]):
        l["n_macro"] = macro_electrons(n, I)
        l["spot_r"] = min(l["spot_r"], 0.4e-6 * case["cross"])  # the laser disc has to fit on the face
    return cfg["targets"], cfg["lasers"], W.run(seed=seed, max_history=400), cfg["I_Wcm2"], counts


def parts(case: dict, seed: int) -> list:
    """(target, laser, run, electrons) of each target of a case."""
    real = in_precision(case)
    if case["kind"] == "emission":
        c = W.config5(case["electrons"])
        p = electrons(case["electrons"], (8, 8, 8), 10e6 * QE / MC2, None, seed, real)
        return [(c["target"], c["laser"], dict(c["run"], seed=seed), p)]
    if case["kind"] == "batch":
        ts, ls, run, I, counts = batch_of(case, seed)
        return [(t, l, dict(run, target_index=i),
                 electrons(counts[i], (t["nx"], t["ny"], t["nz"]), mean_energy(I[i]), l["spot_r"] / t["dx"],
                           seed * 1000 + i, real)) for i, (t, l) in enumerate(zip(ts, ls))]
    t = target_of(case)
    l = laser_of(case, t)
    p = electrons(case["electrons"], (t["nx"], t["ny"], t["nz"]), mean_energy(case["intensity"]),
                  l["spot_r"] / t["dx"], seed, real)
    return [(t, l, run_of(case, seed), p)]


def points(case: dict, seed: int) -> list:
    rng = np.random.default_rng(seed)
    pts = []
    for z in range(case["elements"]):
        for i in range(case["intensities"]):
            f = (i + rng.uniform(0, 0.5)) / max(case["intensities"] - 1, 1)
            pts.append(W.model_point(Z=1.0 + z, I_Wcm2=10.0 ** (20 + 2 * min(f, 1.0))))
    return pts


def prepare(case: dict, seed: int):
    if case["kind"] == "model":
        pts = points(case, seed)
        src = (hpic.hpic_model_in * len(pts))(*[hpic.model_in(m) for m in pts])
        host = torch.frombuffer(bytearray(bytes(src)), dtype=torch.uint8)
        words = ctypes.sizeof(hpic.hpic_model_out) // 8
        return {"case": case, "n": len(pts), "in": host.cuda(),
                "out": torch.zeros(len(pts), words, dtype=torch.float64, device="cuda")}
    prec = hpic.HPIC_FP32_MIXED if case["precision"] == "fp32" else hpic.HPIC_FP64
    each = parts(case, seed)
    if case["kind"] == "batch":
        sim = hpic.Batch([p[0] for p in each], [p[1] for p in each], dict(each[0][2], target_index=0), precision=prec,
                         spare_slots=max(len(p[3]["id"]) for p in each), sort_interval=case["sort"])
        sim.set_tuning(case["blocks"], case["sort"])
        views = sim.targets
    else:
        sim = hpic.Sim(*each[0][:3], precision=prec, sort_interval=case.get("sort", 0))
        views = [sim]
    host = [page_locked(p, t["dx"]) for t, _, _, p in each]
    if case["kind"] != "emission":
        for i, (v, (t, _, _, _)) in enumerate(zip(views, each)):
            for k, g in fields(t, seed * 1000 + i).items():
                v.set_grid(k, g.reshape(-1))
    back = kept = None
    if returns_electrons(case):
        n = room(case, each[0])
        back = page_locked({k: torch.zeros(n, dtype=torch.float64) for k in KEYS + ("id",)}, 1.0)
        kept = {k: torch.zeros(n, dtype=in_precision(case)) for k in KEYS}
    return {"case": case, "sim": sim, "views": views, "host": host, "back": back, "kept": kept}


def in_precision(case: dict) -> torch.dtype:
    return torch.float32 if case["precision"] == "fp32" else torch.float64


def returns_electrons(case: dict) -> bool:
    return case["kind"] == "emission" or bool(case.get("electrons_out"))


def dumped(case: dict) -> list:
    """The grids that a pass reads back: those that last from step to step, and E beside the electrons."""
    if case["kind"] == "emission":
        return []
    return ["T", "B"] + (["E"] if returns_electrons(case) else []) + (["Ti"] if case.get("physics") == "screened" else [])


def single_electrons(case: dict) -> bool:
    """Whether each electron's path can be told: in single precision a last bit turns the scatter frame of
    about one in 1e7 electron-steps, so the paths of large FP32 runs are those of no other run; their
    optical depths (and the fields and energies of all of them) are."""
    return case["precision"] == "fp64" or case["electrons"] <= 5000


# ---------------------------------------------------------------- a pass
def run(state):
    case = state["case"]
    if case["kind"] == "model":
        hpic.hpic_model_device(state["n"], state["in"].data_ptr(), state["out"].data_ptr(),
                               stream=torch.cuda.current_stream().cuda_stream)
        out = state["out"]
        return {"values": out[:, :-1], "steps": out.view(torch.int64)[:, -1]}
    for v, p in zip(state["views"], state["host"]):
        v.set_particles(p)
        if case.get("inject") == "gauss":
            v.set_weights(p["w"])
        v.set_clock(first_step(case), len(p["id"]))
    state["sim"].step(case["steps"])
    kept, out = in_precision(case), []
    for v in state["views"]:
        budget = v.tallies()
        r = {"budget": torch.tensor([budget[k] for k in BUDGET], dtype=kept)}
        for k in dumped(case):
            names = [k + c for c in "xyz"] if k in "EB" else [k]
            r[k] = torch.stack([torch.from_numpy(v.grid(q)).to(kept) for q in names])
        if case.get("spectrum"):
            r["photon_energy"], r["photons"] = [torch.from_numpy(h).to(kept) for h in v.hist()]
        if state["back"] is not None:  # the live ones first, then zeros
            live = v.particles(state["back"])
            n = len(live["id"])
            for k in KEYS if single_electrons(case) else ("tau",):
                state["kept"][k][:n].copy_(torch.from_numpy(live[k]))
                state["kept"][k][n:] = 0
                r["electron_" + k] = state["kept"][k]
            state["back"]["id"][n:] = 0
            r["electron_id"] = state["back"]["id"].view(np.int32)
        out.append(r)
    return out


def room(case: dict, part) -> int:
    """Electrons at the end of a pass, at most: those restored and those that the laser adds."""
    s0, inject = first_step(case), case.get("inject", "none")
    t, l, run = part[:3]
    n = case["electrons"]
    if inject == "flat":
        S = round(l["t_inj"] / run["dt"])
        n += (l["n_macro"] * (s0 + case["steps"])) // S - (l["n_macro"] * s0) // S
    elif inject == "gauss":
        n += case["steps"] * l["per_cell"] * t["ny"] * t["nz"]
    return n


def work(case: dict) -> dict:
    """Bytes and operations of a pass: the electrons and the grid stream through once a step."""
    if case["kind"] == "model":
        n = case["intensities"] * case["elements"]
        return {"bytes": n * 328.0, "flops": n * 2300 * 4 * 90.0}
    real = 4 if case["precision"] == "fp32" else 8
    nodes = 0
    if case["kind"] == "step":
        nodes = (case["nx"] + 1) * (case["ny"] + 1) * (case["nz"] + 1)
    elif case["kind"] == "batch":
        nodes = case["targets"] * (case["cross"] + 1) ** 2 * (0.5 * (case["thin"] + case["thick"]) + 1)
    per_electron, flops = 14 * real + 4, 700.0 if case["kind"] == "emission" else 1210.0
    # E, B and j read, E and B written, T, eta and the drag heat read, T and eta written
    per_node = 15 * real + 5 * 8
    n = case["electrons"]
    return {"bytes": float(case["steps"] * (n * per_electron + nodes * per_node)),
            "flops": float(case["steps"] * (n * flops + nodes * 90))}


# ---------------------------------------------------------------- the method in 64 bits
def philox(step, ids, block, target, seed):
    """Philox4x32-10 of counter (step, id, block, target); the four words as open-interval uniforms."""
    m = 0xFFFFFFFF
    c = [torch.full_like(ids, step & m), ids, torch.full_like(ids, block), torch.full_like(ids, target)]
    k0, k1 = seed & m, (seed >> 32) & m
    for _ in range(10):
        p0, p1 = c[0] * 0xD2511F53, c[2] * 0xCD9E8D57
        c = [((p1 >> 32) & m) ^ c[1] ^ k0, p1 & m, ((p0 >> 32) & m) ^ c[3] ^ k1, p0 & m]
        k0, k1 = (k0 + 0x9E3779B9) & m, (k1 + 0xBB67AE85) & m
    return [((v >> 9).double() + 0.5) / 8388608.0 for v in c]


def kinetic(u):
    u2 = (u * u).sum(0)
    return u2 / (1 + torch.sqrt(1 + u2))


def momentum(e):
    return torch.sqrt(e * (e + 2))


def rotate(d, ct, st, cp, sp):
    sg = torch.where(d[2] >= 0, 1.0, -1.0)
    a = -1 / (sg + d[2])
    b = d[0] * d[1] * a
    e1 = torch.stack([1 + sg * d[0] * d[0] * a, sg * b, -sg * d[0]])
    e2 = torch.stack([b, sg + d[1] * d[1] * a, -d[1]])
    return d * ct + (e1 * cp + e2 * sp) * st


class Solid:
    """Coefficients of one target (Eqs. (5), (B4), (4), (A4)-(A8)), normalised to cells, steps and m_e c^2."""

    def __init__(self, t):
        self.t = t
        self.el = [t] + list(t["extra"])
        self.ne = sum(s["Z"] * s["n_i"] for s in self.el)

    def resistivity(self, T):
        t, kT = self.t, KB * T
        n1 = sum(s["Zstar"] * s["n_i"] for s in self.el)
        n2 = sum(s["Zstar"] ** 2 * s["n_i"] for s in self.el)
        tau = (128 * math.pi * EPS0 ** 2 / (3 * QE ** 4) * math.sqrt(ME / (2 * math.pi)) / (n2 * t["lnLambda"])) * kT ** 1.5
        if t["lambda1"] > 0:
            n0 = sum(s["n_i"] for s in self.el)
            cold = (3 / (4 * math.pi * n0)) ** (1 / 3) * t["lambda1"] * math.sqrt(ME / 3)
            tau = torch.maximum(tau, cold / torch.sqrt(kT))
        return torch.clamp(t["lambda2"] * ME / (n1 * QE ** 2) / tau, max=t["eta_max"])

    def warmed(self, T, rho):
        inv = 0.0
        for s in self.el:
            tp = KB / QE * s["Z"] ** (-4 / 3) * T
            inv = inv + s["Z"] * s["n_i"] / self.ne / (0.3 + 1.2 * tp * (2.2 + tp) / (1.1 + tp) ** 2)
        return T + rho * inv / (self.ne * KB)

    def screening(self, Ti):
        t = self.t
        a_s = 1.4 * A_BOHR * t["Z"] ** (-1 / 3)
        debye = torch.sqrt(EPS0 * KB * Ti / (t["n_i"] * t["Zstar"] ** 2 * QE ** 2))
        return 1 + torch.log(debye / a_s) / math.log(a_s * ME * CL / HBAR) * (t["Zstar"] / t["Z"]) ** 2

    def scatter_log(self, Z):
        return 4 * EPS0 * HPL * CL / (Z ** (1 / 3) * QE ** 2)


def shape_G(u0):
    return 4 / 3 * (-torch.log(u0) - (1 - u0)) + 0.5 * (1 - u0 * u0)


def photon_table(run, dev):
    """ln(eps/k) / ln(eps/k_min) over the electron's energy (rows) and the uniform deviate (columns)."""
    rows, cols = run["table_rows"], run["table_cols"]
    lu0 = (-math.log(run["table_E_max"] / run["k_min"]) * torch.arange(rows, device=dev, dtype=torch.float64) / (rows - 1))[:, None]
    r = torch.linspace(0, 1, cols, device=dev, dtype=torch.float64)[None, :]
    want = r * shape_G(torch.exp(lu0))
    lo, hi = lu0.expand(rows, cols).clone(), torch.zeros(rows, cols, device=dev, dtype=torch.float64)
    for _ in range(80):  # bisection on ln(k/eps)
        y = 0.5 * (lo + hi)
        e, u0 = torch.exp(y), torch.exp(lu0)
        G = 4 / 3 * (y - lu0 - (e - u0)) + 0.5 * (e * e - u0 * u0)
        lo, hi = torch.where(G < want, y, lo), torch.where(G < want, hi, y)
    w = 0.5 * (lo + hi) / lu0
    w[0], w[:, 0], w[:, -1] = 1 - r[0], 1.0, 0.0
    return w


class Exact:
    """One target advanced in 64 bits."""

    def __init__(self, t, l, run, p, grids):
        dev = p["x"].device
        self.t, self.l, self.run, self.s = t, l, run, Solid(t)
        self.n = (t["nx"], t["ny"], t["nz"])
        self.x, self.u = torch.stack([p[k] for k in KEYS[:3]]), torch.stack([p[k] for k in KEYS[3:6]])
        self.tau, self.id = p["tau"].clone(), p["id"].clone()
        dx, dt = t["dx"], run["dt"]
        self.a0 = 8.5e-6 * math.sqrt(l["I0"] * l["lambda"] ** 2)
        self.weighted = l["envelope"] == W.ENV_GAUSS
        w = 1.0
        if not self.weighted and l["n_macro"] > 0:
            w = l["eta_l2e"] * l["I0"] * math.pi * l["spot_r"] ** 2 * l["t_inj"] / (self.a0 * MC2) / l["n_macro"]
        self.w1, self.w = w, p["w"].clone() if self.weighted else torch.full_like(self.tau, w)
        self.cdt = CL * dt / dx
        self.table = photon_table(run, dev)
        self.b = dict.fromkeys(BUDGET, 0.0)
        self.hist = torch.zeros(2, (run["n_E"] + 2) * run["n_theta"], device=dev, dtype=torch.float64)
        self.bounded = not run["physics"] & 64
        if grids:
            g = {k: torch.from_numpy(v).to(dev) for k, v in grids.items()}
            self.E = torch.stack([g[k] for k in ("Ex", "Ey", "Ez")]) * (-QE * dt / (ME * CL))
            self.B = torch.stack([g[k] for k in ("Bx", "By", "Bz")]) * (-QE * dt / ME)
            self.T, self.Ti, self.eta = g["T"], g["Ti"], g["eta"]

    def tally(self, name, v):
        self.b[name] += float(v.sum())

    def lattice(self, axis, half):
        X, n = self.x[axis], self.n[axis]
        q = torch.clamp(X - 0.5, 0, n - 1) if half else X
        i = torch.clamp(torch.floor(q), 0, n - 1)
        return i.long(), q - i

    def corners(self, half):
        """(flat node, weight) of the eight corners; half: the axes on the half-staggered lattice."""
        ax = [self.lattice(a, half[a]) for a in range(3)]
        sy, sz = self.n[0] + 1, (self.n[0] + 1) * (self.n[1] + 1)
        base = ax[0][0] + sy * ax[1][0] + sz * ax[2][0]
        for c in range(8):
            o = (c & 1, c >> 1 & 1, c >> 2)
            w = 1.0
            for a in range(3):
                w = w * (ax[a][1] if o[a] else 1 - ax[a][1])
            yield base + o[0] + sy * o[1] + sz * o[2], w

    def gather(self, G, half):
        flat = G.reshape(-1)
        return sum(flat[q] * w for q, w in self.corners(half))

    def cell(self):
        i = [self.lattice(a, False)[0] for a in range(3)]
        return i[0] + self.n[0] * (i[1] + self.n[1] * i[2])

    def drop(self, keep):
        self.x, self.u = self.x[:, keep], self.u[:, keep]
        self.tau, self.id, self.w = self.tau[keep], self.id[keep], self.w[keep]

    def step(self, step):
        run, t, dt, dx = self.run, self.t, self.run["dt"], self.t["dx"]
        phys, ti, seed = run["physics"], run["target_index"], run["seed"]
        self.b["particle_steps"] += self.x.shape[1]
        eps0 = kinetic(self.u)
        if self.bounded:
            halves = [tuple(a == c for a in range(3)) for c in range(3)]
            E = torch.stack([self.gather(self.E[c], halves[c]) for c in range(3)])
            B = torch.stack([self.gather(self.B[c], tuple(not h for h in halves[c])) for c in range(3)])
            m = self.u + 0.5 * E
            tb = B * (0.5 / torch.sqrt(1 + (m * m).sum(0)))
            s = 2 * tb / (1 + (tb * tb).sum(0))
            q = m + torch.linalg.cross(m, tb, dim=0)
            self.u = m + torch.linalg.cross(q, s, dim=0) + 0.5 * E
            heat = torch.zeros(self.n[0] * self.n[1] * self.n[2], device=self.x.device, dtype=torch.float64)
            F = self.s.screening(self.Ti.reshape(-1))[self.cell()] if phys & 128 else 1.0
        else:
            F = 1.0
        home = self.cell()
        eps = kinetic(self.u)
        self.tally("W_field", self.w * (eps0 - eps))
        # ionisation drag, Eq. (5), and the tracking cut
        cut = run["E_cut"] / MC2
        gam = 1 + eps
        beta = momentum(eps) / gam
        de = 0.0
        for el in self.s.el:
            br = torch.log(eps * MC2 / el["I_ex"]) + 0.5 * torch.log(gam + 1) + 0.909 / gam ** 2 - 0.818 / gam - 0.246
            k = el["Z"] * el["n_i"] * QE ** 4 * dt / (4 * math.pi * EPS0 ** 2 * ME * CL) / MC2
            de = de + k / beta * torch.clamp(br, min=0)
        alive = (eps >= cut) & (eps - de >= cut)
        dep = self.w * torch.where(alive, de, eps)
        eps = torch.where(alive, eps - de, eps)
        self.u = self.u * torch.where(alive, momentum(eps) / torch.sqrt((self.u * self.u).sum(0)), 1.0)
        # Davies scatter, Eq. (B4)
        r = philox(step, self.id, 0, ti, seed)
        un = torch.sqrt((self.u * self.u).sum(0))
        var = 0.0
        for el in self.s.el:
            k = el["Z"] ** 2 * QE ** 4 * el["n_i"] * dt / (2 * math.pi * EPS0 ** 2 * ME ** 2 * CL ** 3)
            var = var + k * torch.sqrt(1 + un * un) / un ** 3 * torch.clamp(torch.log(self.s.scatter_log(el["Z"]) * un), min=0)
        th = torch.sqrt(-2 * torch.log(r[0])) * torch.cos(2 * math.pi * r[1]) * torch.sqrt(var)
        d = rotate(self.u / un, torch.cos(th), torch.sin(th), torch.cos(2 * math.pi * r[2]), torch.sin(2 * math.pi * r[2]))
        self.u = torch.where(alive, un * d, self.u)
        # bremsstrahlung by optical depth (App. B)
        kmin = run["k_min"] / MC2
        rate = sum(QE ** 6 * el["n_i"] * el["Z"] ** 2 * math.log(5.6 * math.pi * EPS0 * HBAR * CL / (el["Z"] ** (1 / 3) * QE ** 2))
                   for el in self.s.el) / (12 * math.pi ** 3 * EPS0 ** 3 * ME * CL ** 3 * HBAR)
        emits = alive & (eps > kmin)
        depth = run["brem_boost"] * rate * CL * dt / MC2 * momentum(eps) / eps * shape_G(kmin / eps) * F
        self.tau = torch.where(emits, self.tau - depth, self.tau)
        at = torch.nonzero(emits & (self.tau <= 0))[:, 0]
        if len(at):
            self.emit(step, at, eps, dep, alive, kmin, cut)
        self.tally("E_drag", dep)
        if self.bounded:
            heat.index_add_(0, home, dep)
        self.b["n_cut"] += float((~alive).sum())
        self.drop(alive)
        ig = 1 / torch.sqrt(1 + (self.u * self.u).sum(0))
        self.x = self.x + self.u * ig * self.cdt
        if self.bounded:
            self.faces(step)
            self.solve(heat)
        self.inject(step)

    def emit(self, step, at, eps, dep, alive, kmin, cut):
        run = self.run
        r = philox(step, self.id[at], 1, run["target_index"], run["seed"])
        e = eps[at]
        lr = torch.log(e / kmin)
        rows, cols = self.table.shape
        L = lr * (rows - 1) / math.log(run["table_E_max"] / run["k_min"])
        i = torch.clamp(torch.floor(L), 0, rows - 2)
        f = torch.clamp(L - i, 0, 1)
        c = r[0] * (cols - 1)
        j = torch.floor(c)
        g, i, j = c - j, i.long(), j.long()
        tab = self.table
        row = [tab[i + a, j] * (1 - g) + tab[i + a, j + 1] * g for a in (0, 1)]
        x = (row[0] * (1 - f) + row[1] * f) * lr
        k = e * torch.exp(-x)
        gam = 1 + e
        a2 = (math.pi * gam) ** 2
        th = torch.sqrt(r[1] * a2 / (1 + a2) / (1 - r[1] + r[1] / (1 + a2))) / gam
        u = self.u[:, at]
        un = torch.sqrt((u * u).sum(0))
        d = rotate(u / un, torch.cos(th), torch.sin(th), torch.cos(2 * math.pi * r[2]), torch.sin(2 * math.pi * r[2]))
        polar = torch.atan2(torch.sqrt(d[1] ** 2 + d[2] ** 2), d[0])
        lo, hi = run["tally_E_min"] / MC2, run["tally_E_max"] / MC2
        bin_e = torch.clamp(1 + torch.floor(run["n_E"] / math.log(hi / lo) * torch.log(k / lo)), 1, run["n_E"])
        bin_e = torch.where(k < lo, 0.0, torch.where(k >= hi, run["n_E"] + 1.0, bin_e))
        col = torch.clamp(torch.floor(polar * run["n_theta"] / math.pi), 0, run["n_theta"] - 1)
        wph = self.w[at] / run["brem_boost"]
        at_bin = (bin_e * run["n_theta"] + col).long()
        self.hist[0].index_add_(0, at_bin, wph * k)
        self.hist[1].index_add_(0, at_bin, wph)
        self.tally("E_xray", wph * k)
        self.tally("E_xray_above", (wph * k)[k >= run["ce_threshold"] / MC2])
        self.b["n_emitted"] += len(at)
        self.tau[at] = -torch.log(1 - r[3])
        ib = 1 / run["brem_boost"]
        left = e * ((1 - ib) - ib * torch.expm1(-x))
        gone = left < cut
        dep[at] += torch.where(gone, self.w[at] * left, 0.0)
        alive[at] = ~gone
        self.u[:, at] = torch.where(gone, u, u * (momentum(left) / un))

    def faces(self, step):
        run = self.run
        for a in range(3):
            L = float(self.n[a])
            out = (self.x[a] < 0) | (self.x[a] > L)
            if not bool(out.any()):
                continue
            e = kinetic(self.u)
            escape = out & (e >= run["kappa_esc"] * self.a0)
            self.tally("E_escaped", (self.w * e)[escape])
            self.b["n_escaped"] += float(escape.sum())
            un = torch.sqrt((self.u * self.u).sum(0))
            un2 = un - run["kappa_tnsa"] * self.a0
            lost = out & ~escape & (un2 <= 0)
            self.tally("E_reflux", (self.w * e)[lost])
            self.b["n_reflux_absorbed"] += float(lost.sum())
            at = torch.nonzero(out & ~escape & ~lost)[:, 0]
            low = self.x[a, at] < 0
            self.x[a, at] = torch.where(low, -self.x[a, at], 2 * L - self.x[a, at])
            d = self.u[:, at] / un[at]
            d[a] = -d[a]
            r = philox(step, self.id[at], 2 + a, run["target_index"], run["seed"])
            xi = run["sigma_dtheta"] * (r[0] - 0.5)
            d = rotate(d, torch.cos(xi), torch.sin(xi), torch.cos(2 * math.pi * r[1]), torch.sin(2 * math.pi * r[1]))
            d[a] = torch.where(low, torch.abs(d[a]), -torch.abs(d[a]))
            self.u[:, at] = un2[at] * d
            self.tally("E_reflux", self.w[at] * (e[at] - kinetic(self.u[:, at])))
            self.b["n_refluxed"] += len(at)
            self.drop(~(escape | lost))

    def solve(self, heat):
        t, run, dt, dx = self.t, self.run, self.run["dt"], self.t["dx"]
        nx, ny, nz = self.n
        J = torch.zeros_like(self.E)
        v = self.w * self.u / torch.sqrt(1 + (self.u * self.u).sum(0))
        for c in range(3):
            flat = J[c].reshape(-1)
            for q, w in self.corners(tuple(a == c for a in range(3))):
                flat.index_add_(0, q, v[c] * w)
        Fc = 1 / (CL * dx * MU0) if run["curlB_term"] else 0.0
        Fj = QE ** 2 * dt / (ME * dx ** 3)
        B, eta, E = self.B, self.eta, torch.zeros_like(self.E)

        def back(G, axis, inner):  # G - its neighbour below along `axis`, on the inner nodes
            return (G - torch.roll(G, 1, 2 - axis))[inner]

        for c in range(3):
            a, b = (c + 1) % 3, (c + 2) % 3
            inner = [slice(1, n) for n in (nz, ny, nx)]
            inner[2 - c] = slice(0, self.n[c])
            inner = tuple(inner)
            curl = back(B[b], a, inner) - back(B[a], b, inner)
            lo = [[slice(0, -1), slice(1, None)], [slice(0, -1), slice(1, None)], [slice(0, -1), slice(1, None)]]
            lo[2 - c] = [slice(None)]
            mean = sum(eta[k, j, i] for k in lo[0] for j in lo[1] for i in lo[2]) / 4
            E[c][inner] = mean * (Fc * curl - Fj * J[c][inner])
        self.E = E

        def fore(G, axis):
            return torch.roll(G, -1, 2 - axis) - G

        for c in range(3):
            a, b = (c + 1) % 3, (c + 2) % 3
            s = [slice(0, n) for n in (nz, ny, nx)]
            s[2 - c] = slice(None)
            s = tuple(s)
            B[c][s] -= self.cdt * (fore(E[b], a) - fore(E[a], b))[s]
        jb2 = 0.0
        for c in range(3):
            a, b = (c + 1) % 3, (c + 2) % 3
            m = J[c] + torch.roll(J[c], -1, 2 - a)
            jb2 = jb2 + (0.25 * (m + torch.roll(m, -1, 2 - b)))[:nz, :ny, :nx] ** 2
        ohm = eta * (QE * CL / dx ** 3) ** 2 * dt * jb2
        self.tally("E_ohmic_grid", ohm * dx ** 3)
        rho = heat.reshape(nz, ny, nx) * MC2 / dx ** 3 + ohm
        self.T = torch.where(rho != 0, self.s.warmed(self.T, rho), self.T)
        if run["physics"] & 256:
            mi, me = t["A_ion"], ME / AMU
            a = (t["Zstar"] ** 2 * QE ** 4 * t["n_i"] * dt * 2 / (3 * (2 * math.pi * KB) ** 1.5) * math.sqrt(me * mi) * t["lnLambda"]
                 / (EPS0 ** 2 * math.sqrt(AMU))) / (self.T * mi + self.Ti * me) ** 1.5
            b, gap = t["Zstar"] * a, self.T - self.Ti
            f = torch.expm1(-(a + b)) / (a + b)
            self.T, self.Ti = self.T + a * gap * f, self.Ti - b * gap * f
        self.eta = self.s.resistivity(self.T)

    def inject(self, step):
        l, run, dx, dt = self.l, self.run, self.t["dx"], self.run["dt"]
        dev, first = self.x.device, self.next_id
        if self.weighted:
            t_pk = 0.5 * l["t_fwhm"] * math.sqrt(math.log(1 / l["g_min"]) / math.log(2))
            gt = math.exp(-4 * math.log(2) * ((step + 0.5) * dt - t_pk) ** 2 / l["t_fwhm"] ** 2)
            y, z = [(torch.arange(n, device=dev, dtype=torch.float64) + 0.5) * dx - l[k] for n, k in ((self.n[1], "spot_y"), (self.n[2], "spot_z"))]
            f = torch.exp(-4 * math.log(2) * (y[None, :] ** 2 + z[:, None] ** 2) / l["r_fwhm"] ** 2)
            kj = torch.nonzero(f >= l["f_min"])
            n = len(kj) * l["per_cell"] if gt >= l["g_min"] else 0
        else:
            S = max(1, round(l["t_inj"] / dt))
            n = l["n_macro"] * (step + 1) // S - l["n_macro"] * step // S if step < S else 0
        if n <= 0:
            return
        ids = torch.arange(first, first + n, device=dev)
        self.next_id += n
        r8, r9 = philox(step, ids, 8, run["target_index"], run["seed"]), philox(step, ids, 9, run["target_index"], run["seed"])
        if self.weighted:
            kj = kj.repeat_interleave(l["per_cell"], 0)
            sfg = torch.sqrt(f[kj[:, 0], kj[:, 1]] * gt)
            mean = self.a0 * sfg
            w = l["I0"] * dx * dx * dt * l["eta_l2e"] / (self.a0 * MC2 * l["per_cell"]) * sfg
            y, z = kj[:, 1] + r8[0], kj[:, 0] + r8[1]
        else:
            rr, mean, w = l["spot_r"] / dx * torch.sqrt(r8[0]), self.a0, torch.full_like(r8[0], self.w1)
            y = l["spot_y"] / dx + rr * torch.cos(2 * math.pi * r8[1])
            z = l["spot_z"] / dx + rr * torch.sin(2 * math.pi * r8[1])
        eps = -mean * torch.log(1 - r8[2])
        omc = torch.full_like(eps, 2 * math.sin(0.5 * l["cone_half"]) ** 2)
        if l["moore_cap"]:
            omc = torch.minimum(omc, 2 / (2 + eps) / (1 + torch.sqrt(eps / (2 + eps))))
        omc = r8[3] * omc
        st, un = torch.sqrt(omc * (2 - omc)), momentum(eps)
        u = torch.stack([un * (1 - omc), un * st * torch.cos(2 * math.pi * r9[0]), un * st * torch.sin(2 * math.pi * r9[0])])
        self.x = torch.cat([self.x, torch.stack([torch.full_like(y, 1e-6), y, z])], 1)
        self.u, self.tau = torch.cat([self.u, u], 1), torch.cat([self.tau, -torch.log(1 - r9[1])])
        self.id, self.w = torch.cat([self.id, ids]), torch.cat([self.w, w])
        self.tally("E_injected", w * eps)
        self.tally("N_injected", w)
        self.b["n_injected"] += n

    def budget(self):
        b = dict(self.b)
        for k in ("E_injected", "W_field", "E_drag", "E_xray", "E_xray_above", "E_escaped", "E_reflux"):
            b[k] *= MC2
        b["E_live"] = float((self.w * kinetic(self.u)).sum()) * MC2
        if self.bounded:
            b["E_B_field"] = float((self.B ** 2).sum()) * (ME / (QE * self.run["dt"])) ** 2 * self.t["dx"] ** 3 / (2 * MU0)
        return np.array([b[k] for k in BUDGET])


def exact(case: dict, seed: int):
    if case["kind"] == "model":
        return model_exact(points(case, seed))
    out = []
    for i, (t, l, run, p) in enumerate(parts(case, seed)):
        grids = fields(t, seed * 1000 + i) if case["kind"] != "emission" else None
        x = Exact(t, l, run, p, grids)
        x.next_id = len(p["id"])
        for s in range(case["steps"]):
            x.step(first_step(case) + s)
        r = {"budget": x.budget()}
        dt = run["dt"]
        if grids:
            have = {"T": x.T[None], "Ti": x.Ti[None], "B": x.B * (-ME / (QE * dt)), "E": x.E * (-ME * CL / (QE * dt))}
            r.update({k: have[k].reshape(have[k].shape[0], -1).cpu() for k in dumped(case)})
        if case.get("spectrum"):
            h = x.hist.reshape(2, run["n_E"] + 2, run["n_theta"]).cpu()
            r["photon_energy"], r["photons"] = h[0] * MC2, h[1]
        if returns_electrons(case):
            n = room(case, (t, l, run))

            def padded(v):
                return torch.cat([v.cpu(), torch.zeros(n - len(v), dtype=v.dtype)])

            if single_electrons(case):
                for a, k in enumerate("xyz"):
                    r["electron_" + k], r["electron_u" + k] = padded(x.x[a] * t["dx"]), padded(x.u[a])
            r["electron_tau"], r["electron_id"] = padded(x.tau), padded(x.id)
        out.append(r)
    return out


def model_exact(pts: list) -> dict:
    """The three-macro-electron estimate (Sec. III.B): RK4 of every set's warm, emitting and escaping band."""
    dev = device()

    def col(k):
        return torch.tensor([float(m[k]) for m in pts], dtype=torch.float64, device=dev)

    c = {k: col(k) for k in pts[0]}
    a0 = 8.5e-6 * torch.sqrt(c["I0"] * c["lambda"] ** 2)
    T = a0 * MC2 * c["mean_sqrt_fg"]
    Lrad = torch.log(5.6 * math.pi * EPS0 * HBAR * CL / (c["Z"] ** (1 / 3) * QE ** 2))
    Kb = QE ** 6 / (12 * math.pi ** 3 * EPS0 ** 3 * ME * CL ** 3 * HBAR) * c["n_i"] * c["Z"] ** 2 * Lrad
    Ki = c["Z"] * c["n_i"] * QE ** 4 / (4 * math.pi * EPS0 ** 2 * ME * CL ** 2)
    St = 3 * c["kappa_tnsa"] * a0 * MC2 / (c["Lx"] + c["Ly"] + c["Lz"])
    r, tc = 0.5 * c["r_fwhm"], torch.tan(c["theta_c"])
    Fc = QE ** 2 * c["eta_avg"] * c["I0"] * c["mean_fg"] * r * r * c["eta_l2e"] / T
    N = c["I0"] * c["mean_fg"] * (math.pi * c["r_fwhm"] ** 2 / 4) * (c["t_fwhm"] * math.sqrt(math.log(10) / math.log(2))) * c["eta_l2e"] / T
    esc, th = c["kappa_esc"] * a0 * MC2, c["eps_th"]
    n = len(pts)
    E, bands, steps = torch.zeros(n, 8, dtype=torch.float64, device=dev), [], torch.zeros(n, dtype=torch.int64, device=dev)
    inf = torch.full_like(esc, math.inf)
    for b, (lo, hi) in enumerate(((torch.zeros_like(esc), torch.minimum(th, esc)), (th, esc), (esc, inf))):
        top = torch.where(torch.isinf(hi), 0.0, torch.exp(-hi / T))
        topE = torch.where(torch.isinf(hi), 0.0, (hi + T) * torch.exp(-hi / T))
        nb = torch.where(hi > lo, N * (torch.exp(-lo / T) - top), 0.0)
        Eb = torch.where(hi > lo, N * ((lo + T) * torch.exp(-lo / T) - topE), 0.0)
        on = nb > 0
        eps = torch.where(on, Eb / nb, 0.0)
        first, x, acc, at = eps.clone(), torch.zeros_like(eps), torch.zeros(n, 6, dtype=torch.float64, device=dev), torch.nonzero(on)[:, 0]

        def rates(e, z):
            gam = 1 + e / MC2
            ig = 1 / gam
            br = torch.log(torch.clamp(e, min=1e-300) / c["I_ex"][at]) + 0.5 * torch.log(torch.clamp(gam + 1, min=1e-300)) + 0.909 * ig * ig - 0.818 * ig - 0.246
            ion = torch.where((e > 0) & (br > 0), Ki[at] / (1 - ig * ig) * br, 0.0)
            above = torch.where(e > th[at], Kb[at] * (1 + (e - th[at]) / MC2), 0.0)
            return torch.stack([Kb[at] * gam, ion, St[at], Fc[at] / (z * tc[at] + r[at]) ** 2, above], 1)

        while len(at):  # the sets still under way
            e, z = eps[at], x[at]
            end = (z >= c["Lx"][at]) if b == 2 else (e <= c["E_stop"][at])
            acc[at[end], 5 if b == 2 else 1] += e[end]
            at = at[~end]
            at = at[eps[at] > 0]
            if not len(at):
                break
            e, z = eps[at], x[at]
            k1 = rates(e, z)
            t1 = k1[:, :4].sum(1)
            h = torch.minimum(c["rel_step"][at] * e / t1, c["rel_step"][at] * (z + r[at] / tc[at]))
            if b == 2:
                h = torch.where(z + h > c["Lx"][at], c["Lx"][at] - z, h)
            k2 = rates(e - 0.5 * h * t1, z + 0.5 * h)
            k3 = rates(e - 0.5 * h * k2[:, :4].sum(1), z + 0.5 * h)
            k4 = rates(e - h * k3[:, :4].sum(1), z + h)
            steps[at] += 1
            d = (h / 6)[:, None] * (k1 + 2 * k2 + 2 * k3 + k4)
            de = d[:, :4].sum(1)
            stop = de >= e
            share = torch.where(stop, e / de, 1.0)
            acc[at, :5] += d * share[:, None]
            x[at] = z + h * share
            eps[at] = e - de
            at = at[~stop]
        E[:, 0] += Eb
        E[:, 1:7] += nb[:, None] * acc
        bands.append((nb, first, x))
    cols = [E, N[:, None], a0[:, None]] + [torch.stack([b[q] for b in bands], 1) for q in range(3)]
    return {"values": torch.cat(cols, 1).cpu(), "steps": steps.cpu()}
