"""Workloads of this framework for timing, with their exact answers.

Each case is one call sequence of a user's program through the package's
public entry points: 3D near-field runs (``Simulation``), their gradients
(``adjoint.TraceModel``), uneven batches (``Batch``), the 2D axisymmetric
solver (``Cylinder``), the lattice surrogate's training step and serving call
(``surrogate.Lattice``), one layer of the MLP surrogate (``sur_*``) and the
spectra of detector traces (``trace_spectrum``).  Sizes are those of
``workloads.py``, ``bench.py`` and the tests, and ragged ones of the same
ranges.

``exact`` restates each of them in 64-bit torch on plain arrays, without the
package.
"""
from __future__ import annotations

import ctypes
import math

import numpy as np
import torch

C0 = 299792458.0
MU0 = 1.25663706212e-6
EPS_R = 3.17                       # ice
PEC, MUR, CPML = 0, 1, 2


def listed():
    return [
        # the smallest 3D run: one shower in a 96^3 box with Mur walls, 8 detectors
        # (the parity workload at its own step count); latency and launches count
        {"name": "fdtd_mur_96", "kind": "fdtd", "nx": 96, "ny": 96, "nz": 96, "boundary": MUR, "npml": 0,
         "dx": 0.02, "half_cell": False, "steps": 400, "probes": 8, "lateral": 4, "layout": "sphere"},
        # the surrogate's data generation (2048 steps a run), the part in which the shower
        # crosses the grid: 128 x 128 x 512 cells, CPML, half a cell per step, every antenna
        # of the lattice (31 radii x 113 bins)
        {"name": "fdtd_data_128x512", "kind": "fdtd", "nx": 128, "ny": 128, "nz": 512, "boundary": CPML, "npml": 10,
         "dx": 0.02, "half_cell": True, "steps": 900, "probes": 3503, "lateral": 15, "layout": "lattice"},
        # a stretch of the headline run (4000 steps in all): 384 x 384 x 1536, 10-cell CPML, 64 detectors
        {"name": "fdtd_greisen_384", "kind": "fdtd", "nx": 384, "ny": 384, "nz": 1536, "boundary": CPML, "npml": 10,
         "dx": 0.02, "half_cell": False, "steps": 120, "probes": 64, "lateral": 15, "layout": "cylinder"},
        # a stretch of the largest run (6000 steps in all): 640 x 640 x 2048, 12-cell CPML, 256 detectors
        {"name": "fdtd_gh_640", "kind": "fdtd", "nx": 640, "ny": 640, "nz": 2048, "boundary": CPML, "npml": 12,
         "dx": 0.03, "half_cell": False, "steps": 60, "probes": 256, "lateral": 10, "layout": "cylinder"},
        # one gradient of an inversion: forward and backward through torch autograd on
        # the 256 x 256 x 512 closed box, 256-bin charge table, 64 detectors
        {"name": "adjoint_pec_256", "kind": "adjoint", "nx": 256, "ny": 256, "nz": 512, "boundary": PEC, "npml": 0,
         "steps": 120, "probes": 64, "bins": 256, "lateral": 4},
        # independent showers on uneven grids of 64^3 .. 256 x 256 x 512 advanced as one batch
        {"name": "batch_uneven_24", "kind": "batch", "grids": 24, "lo": 64, "hi": 256, "hi_z": 512, "steps": 60,
         "probes": 8, "sizes": 6006},
        # the paper's own 2D formulation, a small grid of its Table I over its whole run
        {"name": "cyl_512", "kind": "cyl", "nr": 512, "nz": 512, "boundary": MUR, "steps": 512, "probes": 64},
        # and its largest grid
        {"name": "cyl_8192", "kind": "cyl", "nr": 8192, "nz": 8192, "boundary": MUR, "steps": 256, "probes": 64},
        # one optimiser step of the lattice surrogate in mid-training: 1024 (shower, antenna) pairs
        {"name": "lattice_train_1024", "kind": "lattice_train", "batch": 1024, "K": 128, "NR": 31, "m_lo": 3,
         "m_hi": 115, "T": 1024, "S": 4, "relative": False},
        # serving it: 64 showers at 64 antennas each (batch 4096)
        {"name": "lattice_serve_64x64", "kind": "lattice_serve", "profiles": 64, "antennas": 64, "K": 128, "NR": 31,
         "m_lo": 3, "m_hi": 115, "T": 1024, "S": 4},
        # one hidden layer of the MLP surrogate, forward and backward: 32 pairs x 128 bins as rows
        {"name": "mlp_layer_4096x1024", "kind": "mlp_layer", "rows": 4096, "fan_in": 1024, "fan_out": 1024,
         "relu": True},
        # spectra of the 64 detectors of the largest 2D run at 1024 frequencies
        {"name": "spectrum_64x8204", "kind": "spectrum", "traces": 64, "samples": 8204, "freqs": 1024,
         "comps": 2, "gated": True, "taper": 0.2},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["fdtd", "fdtd", "fdtd", "adjoint", "batch", "cyl", "cyl", "lattice_train", "lattice_serve",
                       "mlp_layer", "spectrum"])
    if kind == "fdtd":
        b = rng.choice([MUR, CPML, CPML, PEC])
        nx, ny = _log(rng, 48, 400), _log(rng, 48, 400)
        nz = _log(rng, 48, 1200)
        cells = nx * ny * nz
        P = rng.choice([8, 10, 12]) if b == CPML else 0
        # while the shower is in the grid (about half a cell per step)
        steps = max(24, min(400, int(1.5e10 / cells), int(1.6 * (nz - 2 * P - 8))))
        return {"kind": "fdtd", "nx": nx, "ny": ny, "nz": nz, "boundary": b, "npml": P, "dx": rng.choice([0.02, 0.03]),
                "half_cell": rng.random() < 0.25, "steps": steps + rng.randrange(2),
                "probes": rng.choice([1, 8, 64, 200]), "lateral": rng.choice([3, 4, 8]), "layout": "cylinder"}
    if kind == "adjoint":
        b = rng.choice([PEC, CPML, MUR])
        return {"kind": "adjoint", "nx": _log(rng, 48, 200), "ny": _log(rng, 48, 200), "nz": _log(rng, 64, 400),
                "boundary": b, "npml": 8 if b == CPML else 0, "steps": rng.randrange(60, 121),
                "probes": rng.choice([4, 33, 64]), "bins": rng.choice([64, 128, 256]), "lateral": rng.choice([3, 4])}
    if kind == "batch":
        small = rng.random() < 0.5
        return {"kind": "batch", "grids": rng.randrange(8, 40) if small else rng.randrange(4, 16),
                "lo": 32 if small else 64, "hi": 96 if small else 200, "hi_z": 96 if small else 400,
                "steps": rng.randrange(40, 80), "probes": 8, "sizes": rng.randrange(1 << 20)}
    if kind == "cyl":
        nr, nz = _log(rng, 200, 6000), _log(rng, 200, 6000)
        return {"kind": "cyl", "nr": nr, "nz": nz, "boundary": rng.choice([MUR, MUR, PEC]),
                "steps": rng.randrange(120, 400), "probes": rng.choice([1, 16, 64])}
    if kind == "lattice_train":
        return {"kind": "lattice_train", "batch": _log(rng, 100, 3000), "K": rng.choice([64, 100, 128]),
                "NR": rng.choice([7, 16, 31]), "m_lo": rng.choice([0, 3]), "m_hi": rng.choice([57, 90, 115]),
                "T": rng.choice([500, 512, 1024]), "S": 4, "relative": rng.random() < 0.5}
    if kind == "lattice_serve":
        return {"kind": "lattice_serve", "profiles": _log(rng, 1, 1024), "antennas": _log(rng, 1, 256),
                "K": rng.choice([64, 100, 128]), "NR": 31, "m_lo": 3, "m_hi": 115,
                "T": rng.choice([500, 512, 1024]), "S": 4}
    if kind == "mlp_layer":
        return {"kind": "mlp_layer", "rows": 128 * _log(rng, 2, 64), "fan_in": rng.choice([64, 256, 512, 1024]),
                "fan_out": rng.choice([256, 512, 1024, 2048]), "relu": rng.random() < 0.7}
    return {"kind": "spectrum", "traces": _log(rng, 1, 200), "samples": _log(rng, 200, 40000),
            "freqs": _log(rng, 1, 1500), "comps": rng.choice([1, 2, 3]), "gated": rng.random() < 0.5,
            "taper": rng.choice([0.0, 0.2])}


def work(case):
    k = case["kind"]
    if k in ("fdtd", "adjoint"):
        cells = case["nx"] * case["ny"] * case["nz"]
        nodes = (case["nx"] + 1) * (case["ny"] + 1) * (case["nz"] + 1)
        upd = cells * case["steps"] * (2 if k == "adjoint" else 1)
        traces = 8 * case["probes"] * case["steps"]
        return {"bytes": traces + (24 * nodes if k == "fdtd" else 2 * traces), "flops": 30.0 * upd}
    if k == "batch":
        dims = _batch_dims(case)
        return {"bytes": 24.0 * sum((a + 1) * (b + 1) * (c + 1) for a, b, c in dims),
                "flops": 30.0 * case["steps"] * sum(a * b * c for a, b, c in dims)}
    if k == "cyl":
        cells = case["nr"] * case["nz"]
        return {"bytes": 12.0 * cells + 8 * case["probes"] * case["steps"], "flops": 15.0 * cells * case["steps"]}
    if k == "lattice_train":
        B, K, T = case["batch"], case["K"], case["T"]
        n = case["NR"] * (case["m_hi"] - case["m_lo"] + K) * T
        return {"bytes": 4.0 * (6 * n + B * (T + K)), "flops": 4.0 * B * K * T + 12.0 * n}
    if k == "lattice_serve":
        P, A, K, T = case["profiles"], case["antennas"], case["K"], case["T"]
        return {"bytes": 4.0 * (A * P * T + P * K) + 4.0 * min(A, case["NR"]) * K * T, "flops": 6.0 * A * P * T * K}
    if k == "mlp_layer":
        M, K, N = case["rows"], case["fan_in"], case["fan_out"]
        return {"bytes": 4.0 * (2 * M * N + 3 * M * K + N * K) + 2.0 * (2 * M * N + 2 * M * K + 2 * N * K),
                "flops": 6.0 * M * N * K}
    n = case["traces"] * case["samples"]
    return {"bytes": 4.0 * n * case["comps"] + 8.0 * case["traces"] * case["freqs"],
            "flops": 4.0 * n * case["freqs"]}


# ---- inputs (host arrays from the seed alone) ---------------------------------------

def _lateral(L, sigma):
    a = np.arange(-L, L + 1)
    w = np.exp(-(a[None, :] ** 2 + a[:, None] ** 2) / (2.0 * sigma * sigma))
    return np.ascontiguousarray((w / w.sum()).ravel())


def _time_step(dx, half_cell=False, dims=3):
    return dx / (2.0 * C0) if half_cell else 0.5 * dx * math.sqrt(EPS_R) / (C0 * math.sqrt(float(dims)))


def _fdtd_inputs(case, seed):
    """Charge table, lateral weights and detector positions of a 3D run."""
    rng = np.random.default_rng(seed)
    nx, ny, nz, P, dx = case["nx"], case["ny"], case["nz"], case["npml"], case["dx"]
    dt = _time_step(dx, case["half_cell"])
    z0 = (P + 4) * dx
    if case["half_cell"]:
        bin_dz = 4 * dx
        n_bins = max(2, min(128, (nz - 2 * P) // 4 - 1))
    else:
        bin_dz = dx / 4.0
        n_bins = 4 * (nz - 2 * P - 4)
    z = z0 + bin_dz * np.arange(n_bins)
    # a sum of subshowers that start within the run's reach, so that charge flows in it
    reach = min(nz * dx - 2 * z0, C0 * dt * case["steps"])
    q = np.zeros(n_bins)
    for _ in range(int(rng.integers(2, 5))):
        start = z0 - rng.uniform(0.02, 0.3)
        rise = rng.uniform(0.2, 0.8) * max(reach, 0.3)
        lam = rise / rng.uniform(2.0, 5.0)
        x = np.maximum(z - start, 0.0)
        q -= 1.6e-20 * 10.0 ** rng.uniform(8.0, 9.0) * (x / rise) ** (rise / lam) * np.exp((rise - x) / lam)
    L = case["lateral"]
    w = _lateral(L, 0.3 * L)
    lo = P + 1 if case["boundary"] == CPML else 1
    ic, jc = nx // 2, ny // 2
    n = case["probes"]
    if case["layout"] == "lattice":
        i, m = np.meshgrid(np.arange(15, 46), np.arange(3, 116), indexing="ij")
        ijk = np.stack([ic + i.ravel(), np.full(i.size, jc), (P + 4) + 4 * m.ravel()], 1)[:n]
    elif case["layout"] == "sphere":
        R, th, ph = rng.uniform(0.16, 0.46, n) * min(nx, ny, nz), np.radians(rng.uniform(30, 150, n)), rng.uniform(0, 2 * np.pi, n)
        ijk = np.stack([ic + R * np.sin(th) * np.cos(ph), jc + R * np.sin(th) * np.sin(ph), nz // 2 + R * np.cos(th)], 1)
    else:
        # where the shower's field arrives within the run
        travel = min(reach, C0 * dt * case["steps"]) / dx
        R, ph = rng.uniform(0.1, 1.0, n) * min(min(nx, ny) // 2 - lo - 1, 3 + 0.2 * travel), rng.uniform(0, 2 * np.pi, n)
        ijk = np.stack([ic + R * np.cos(ph), jc + R * np.sin(ph), z0 / dx + rng.uniform(0.0, 0.55, n) * travel], 1)
    ijk = np.clip(np.round(ijk).astype(np.int64), lo, np.array([nx, ny, nz]) - lo)
    return {"q": q, "z0": z0, "bin_dz": bin_dz, "w": w, "L": L, "ijk": ijk, "dt": dt}


def _adjoint_inputs(case, seed):
    """Charge tables (first guess and truth) and detectors of an inversion."""
    rng = np.random.default_rng(seed)
    nx, ny, nz, P, dx = case["nx"], case["ny"], case["nz"], case["npml"], 0.02
    dt = _time_step(dx)
    n_bins, z0 = case["bins"], (P + 3) * dx
    reach = min((nz - 2 * P - 8) * dx, C0 * dt * case["steps"])
    bin_dz = max(reach, 0.4) / (n_bins - 1)
    z = z0 + bin_dz * np.arange(n_bins)
    tabs = []
    for _ in range(2):
        zp, l = z0 + rng.uniform(0.3, 0.7) * reach, rng.uniform(0.15, 0.35) * reach
        tabs.append((-1e-9 * rng.uniform(0.5, 1.5) * np.exp(-0.5 * ((z - zp) / l) ** 2)).astype(np.float32))
    lo = P + 1 if case["boundary"] == CPML else 1
    n = case["probes"]
    R, ph = rng.uniform(0.1, 1.0, n) * min(min(nx, ny) // 2 - lo - 1, 3 + 0.25 * reach / dx), rng.uniform(0, 2 * np.pi, n)
    ijk = np.stack([nx // 2 + R * np.cos(ph), ny // 2 + R * np.sin(ph), z0 / dx + rng.uniform(0.0, 0.6, n) * reach / dx], 1)
    ijk = np.clip(np.round(ijk).astype(np.int64), lo, np.array([nx, ny, nz]) - lo)
    return {"q": tabs[0], "q_true": tabs[1], "z0": z0, "bin_dz": bin_dz, "w": _lateral(case["lateral"], 1.0),
            "L": case["lateral"], "ijk": ijk, "dt": dt}


def _batch_dims(case):
    r = np.random.default_rng(case["sizes"])
    return [(int(r.integers(case["lo"], case["hi"] + 1)), int(r.integers(case["lo"], case["hi"] + 1)),
             int(r.integers(case["lo"], case["hi_z"] + 1))) for _ in range(case["grids"])]


def _batch_inputs(case, seed):
    rng = np.random.default_rng(seed)
    dx, out = 0.02, []
    dt = _time_step(dx)
    for nx, ny, nz in _batch_dims(case):
        n_bins = 128
        bin_dz = nz * dx / (n_bins - 1)
        reach = min(nz * dx, C0 * dt * case["steps"])
        z = bin_dz * np.arange(n_bins)
        q = -1e-9 * np.exp(-0.5 * ((z - rng.uniform(0.3, 0.7) * reach) / (rng.uniform(0.15, 0.4) * reach)) ** 2)
        n = case["probes"]
        R, ph = rng.uniform(0.1, 0.4, n) * min(nx, ny), rng.uniform(0, 2 * np.pi, n)
        ijk = np.stack([nx // 2 + R * np.cos(ph), ny // 2 + R * np.sin(ph),
                        rng.uniform(0.1, min(0.9, reach / (nz * dx)) + 0.05, n) * nz], 1)
        ijk = np.clip(np.round(ijk).astype(np.int64), 1, np.array([nx, ny, nz]) - 1)
        out.append({"nx": nx, "ny": ny, "nz": nz, "q": q, "z0": 0.0, "bin_dz": bin_dz, "w": _lateral(3, 1.0), "L": 3,
                    "ijk": ijk, "dt": dt})
    return out


def _cyl_inputs(case, seed):
    """The paper's Gaussian shower model on an (r, z) grid: 256-bin table,
    ring weights of a radial Gaussian, detectors about the maximum."""
    rng = np.random.default_rng(seed)
    nr, nz = case["nr"], case["nz"]
    d = 40.96 / max(nr, nz)
    dt = _time_step(d, dims=2)
    reach = min(nz * d, C0 * dt * case["steps"])
    z0 = 0.02 * nz * d
    n_bins = 256
    bin_dz = max(0.7 * reach, 8 * d) / (n_bins - 1)
    z = bin_dz * np.arange(n_bins)
    q = -1e-9 * np.exp(-0.5 * ((z - rng.uniform(0.3, 0.6) * z[-1]) / (rng.uniform(0.12, 0.25) * z[-1])) ** 2)
    sig = 0.05
    n_rings = max(1, min(nr, int(math.ceil(3 * sig / d)) + 1))
    edge = (np.arange(n_rings) + 0.5) * d
    inside = -np.expm1(-0.5 * (edge / sig) ** 2)
    w = np.diff(inside, prepend=0.0)
    w /= w.sum()
    n = case["probes"]
    ij = np.stack([np.minimum(nr - 1, rng.uniform(0.0, 0.2, n) * reach / d),
                   np.clip((z0 + rng.uniform(0.0, 0.5, n) * reach) / d, 2, nz - 2)], 1)
    return {"q": q, "z0": z0, "bin_dz": bin_dz, "w": w, "ij": ij.astype(np.int64), "d": d, "dt": dt}


def _profiles(gen, n, K):
    """Charge profiles [n, K] as the data generation draws them: one
    Gaisser-Hillas shower each, coulombs per bin."""
    dev = "cuda"
    u = torch.rand(n, 4, generator=gen, device=dev, dtype=torch.float64)
    z = torch.arange(K, device=dev, dtype=torch.float64)[None, :] * 0.08
    start, rise, lam = 0.4 + 1.6 * u[:, :1], 1.0 + 2.5 * u[:, 1:2], 0.25 + 0.35 * u[:, 2:3]
    x = (z - start).clamp_min(0.0)
    q = (x / rise) ** (rise / lam) * torch.exp((rise - x) / lam)
    return (-3.2e-20 * 10.0 ** (8.0 + u[:, 3:4]) * q).float().contiguous()


def _lattice_inputs(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    K, NR, T = case["K"], case["NR"], case["T"]
    D = case["m_hi"] - case["m_lo"] + K
    f = lambda *s: torch.randn(*s, generator=gen, device="cuda")
    # bipolar pulses about a retarded time that grows with the offset
    t = torch.arange(T, device="cuda", dtype=torch.float32)
    t0 = (40.0 + 4.0 * (torch.arange(D, device="cuda") - K).abs())[None, :, None] + 3.0 * torch.arange(NR, device="cuda")[:, None, None]
    u = (t[None, None, :] - t0) / (6.0 + 4.0 * torch.rand(NR, D, 1, generator=gen, device="cuda"))
    G = -u * torch.exp(-0.5 * u * u) + 0.02 * f(NR, D, T)
    n = case.get("batch") or case["antennas"]
    ant = torch.stack([torch.randint(0, NR, (n,), generator=gen, device="cuda"),
                       torch.randint(case["m_lo"], case["m_hi"] + 1, (n,), generator=gen, device="cuda")], 1)
    out = {"G": G.contiguous(), "ant": ant.int().contiguous(), "c_out": 2.5e9,
           "q": _profiles(gen, case.get("batch") or case["profiles"], K)}
    if "batch" in case:
        out["m"] = 1e-4 * f(NR, D, T)
        out["v"] = (1e-4 * f(NR, D, T)) ** 2 + 1e-10
        peak = out["q"].abs().amax(1, keepdim=True)
        uu = (t[None, :] - 300.0 * torch.rand(n, 1, generator=gen, device="cuda")) / 9.0
        out["trace"] = (2.5e9 * peak * (-uu * torch.exp(-0.5 * uu * uu) + 0.05 * f(n, T))).contiguous()
    return out


def _mlp_inputs(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    M, K, N = case["rows"], case["fan_in"], case["fan_out"]
    f = lambda *s: torch.randn(*s, generator=gen, device="cuda")
    h = f(M, K).clamp_min(0.0)                    # activations of the layer before (ReLU)
    dz = 1e-3 * f(M, N) * (torch.rand(M, N, generator=gen, device="cuda") < 0.5)
    w = f(N, K) * math.sqrt(2.0 / K)
    return {"h": h, "hb": h.bfloat16(), "wb": w.bfloat16(), "bias": 0.1 * f(N), "dz": dz, "dzb": dz.bfloat16()}


def _spectrum_inputs(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    rng = np.random.default_rng(seed)
    n, T, c = case["traces"], case["samples"], case["comps"]
    t = torch.arange(T, device="cuda", dtype=torch.float32)[None, :, None]
    at = T * (0.2 + 0.6 * torch.rand(n, 1, c, generator=gen, device="cuda"))
    u = (t - at) / (3.0 + 0.02 * T * torch.rand(n, 1, c, generator=gen, device="cuda"))
    x = (-u * torch.exp(-0.5 * u * u) + 0.01 * torch.randn(n, T, c, generator=gen, device="cuda")).contiguous()
    dt = 1.05e-11
    freqs = np.sort(rng.uniform(5e7, 2e9, case["freqs"]))
    th = np.radians(rng.uniform(30.0, 90.0, n))
    coef = np.zeros((n, c))
    coef[:, 0] = -np.sin(th) if c > 1 else 1.0
    if c > 1:
        coef[:, 1] = np.cos(th)
    gate = None
    if case["gated"]:
        first = rng.integers(0, T // 4 + 1, n)
        gate = np.stack([first, np.minimum(T - first, rng.integers(T // 3, T + 1, n))], 1).astype(np.int32)
    return {"x": x, "dt": dt, "freqs": freqs, "coef": coef, "gate": gate}


# ---- what a user's program has in hand -------------------------------------------------

def prepare(case, seed):
    import paper_1001_5341_gb300 as fd
    k = case["kind"]
    new = lambda *s, dtype=torch.float32: torch.empty(s, dtype=dtype, device="cuda")
    if k == "fdtd":
        p = _fdtd_inputs(case, seed)
        sim = fd.Simulation(case["nx"], case["ny"], case["nz"], case["dx"], p["dt"], EPS_R, case["boundary"], case["npml"])
        sim.set_probes(p["ijk"] * case["dx"], case["steps"])
        return {"kind": k, "sim": sim, "in": p, "steps": case["steps"],
                "trace": new(case["probes"], case["steps"], 2), "E": new(3, *sim.shape), "H": new(3, *sim.shape)}
    if k == "adjoint":
        from paper_1001_5341_gb300.adjoint import TraceModel
        p = _adjoint_inputs(case, seed)
        sim = fd.Simulation(case["nx"], case["ny"], case["nz"], 0.02, p["dt"], EPS_R, case["boundary"], case["npml"])
        sim.set_probes(p["ijk"] * 0.02, case["steps"])
        model = TraceModel(sim, p["z0"], p["bin_dz"], C0, p["w"], p["L"], case["steps"])
        with torch.no_grad():
            target = model(torch.tensor(p["q_true"], device="cuda"))
        return {"kind": k, "model": model, "target": target, "q": torch.tensor(p["q"], device="cuda", requires_grad=True)}
    if k == "batch":
        sims, cells = [], 0
        for p in _batch_inputs(case, seed):
            sim = fd.Simulation(p["nx"], p["ny"], p["nz"], 0.02, p["dt"], EPS_R, MUR)
            sim.set_shower(p["q"], p["z0"], p["bin_dz"], C0, p["w"], p["L"])
            sim.set_probes(p["ijk"] * 0.02, 1000)   # room for the tuner's trial steps
            sims.append(sim)
            cells += math.prod(sim.shape)
        batch = fd.Batch(sims)
        batch.tune(trial_steps=2)
        return {"kind": k, "batch": batch, "sims": sims, "steps": case["steps"], "E": new(3, cells), "H": new(3, cells),
                "trace": new(len(sims), case["probes"], sims[0].max_steps, 2)}
    if k == "cyl":
        p = _cyl_inputs(case, seed)
        cyl = fd.Cylinder(case["nr"], case["nz"], p["d"], p["dt"], EPS_R, case["boundary"])
        cyl.set_shower(p["q"], p["z0"], p["bin_dz"], C0, p["w"])
        cyl.set_probes(p["ij"] * p["d"], case["steps"] + 800)          # room for the tuner's trial steps
        cyl.tune(2)
        return {"kind": k, "cyl": cyl, "steps": case["steps"], "trace": new(case["probes"], cyl.max_steps, 2),
                "fields": [new(*cyl.shape(c)) for c in range(3)]}
    if k in ("lattice_train", "lattice_serve"):
        from paper_1001_5341_gb300 import surrogate as S
        p = _lattice_inputs(case, seed)
        geo = S.LatticeGeometry(K=case["K"], NR=case["NR"], m_lo=case["m_lo"], m_hi=case["m_hi"], T=case["T"],
                                S=case["S"], J=case["S"])
        net = S.Lattice(geo, c_out=p["c_out"])
        net.G.copy_(p["G"])
        if k == "lattice_train":
            net.m.copy_(p["m"])
            net.v.copy_(p["v"])
            net.t = 5000
            return {"kind": k, "net": net, "q": p["q"], "ant": p["ant"], "trace": p["trace"], "relative": case["relative"]}
        net.split()
        return {"kind": k, "net": net, "q": p["q"], "ant": p["ant"]}
    if k == "mlp_layer":
        p = _mlp_inputs(case, seed)
        M, K, N = case["rows"], case["fan_in"], case["fan_out"]
        p.update(kind=k, y=new(M, N), yb=new(M, N, dtype=torch.bfloat16), dw=new(N, K), db=new(N), dh=new(M, K),
                 dzp=new(M, K), dzpb=new(M, K, dtype=torch.bfloat16), relu=int(case["relu"]))
        return p
    p = _spectrum_inputs(case, seed)
    p.update(kind=k, taper=case["taper"])
    return p


# ---- one pass ------------------------------------------------------------------------

def _ptr(t):
    return ctypes.c_void_p(t.data_ptr())


def run(s):
    import paper_1001_5341_gb300 as fd
    k = s["kind"]
    if k == "fdtd":
        sim, p = s["sim"], s["in"]
        sim.reset()
        sim.set_shower(p["q"], p["z0"], p["bin_dz"], C0, p["w"], p["L"])
        sim.step(s["steps"])
        sim.probes(out=s["trace"])
        for c in range(3):
            sim.field(c, out=s["E"][c])
            sim.field(c + 3, out=s["H"][c])
        return [s["trace"], s["E"], s["H"]]
    if k == "adjoint":
        s["q"].grad = None
        y = s["model"](s["q"])
        r = y - s["target"]
        (0.5 * (r * r).sum()).backward()
        return [y.detach(), s["q"].grad]
    if k == "batch":
        for sim in s["sims"]:
            sim.reset()
        s["batch"].step(s["steps"])
        s["batch"].sync()
        at = 0
        for n, sim in enumerate(s["sims"]):
            sim.probes(out=s["trace"][n])
            cells = math.prod(sim.shape)
            for c in range(3):
                sim.field(c, out=s["E"][c, at:at + cells])
                sim.field(c + 3, out=s["H"][c, at:at + cells])
            at += cells
        return [s["trace"], s["E"], s["H"]]
    if k == "cyl":
        cyl = s["cyl"]
        cyl.reset()
        cyl.step(s["steps"])
        cyl.probes(out=s["trace"])
        for c in range(3):
            cyl.field(c, out=s["fields"][c])
        return [s["trace"]] + s["fields"]
    if k == "lattice_train":
        net = s["net"]
        loss = net.train_batch(s["q"], s["ant"], s["trace"], 1e-3, relative=s["relative"])
        return [loss, net.G, net.m, net.v]
    if k == "lattice_serve":
        return s["net"].predict_grid(s["q"], s["ant"])
    if k == "mlp_layer":
        M, K = s["h"].shape
        N = s["wb"].shape[0]
        st = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
        # forward: y = [relu](h W^T + b), with the bf16 copy the next layer reads
        fd.check(fd.sur_gemm_bf16(_ptr(s["hb"]), K, 1, _ptr(s["wb"]), K, 1, _ptr(s["y"]), N, _ptr(s["yb"]), M, N, K,
                                  _ptr(s["bias"]), s["relu"], 0, st))
        # backward from dz: dW = dz^T h, db, dh = dz W, and through the ReLU of the layer before
        fd.check(fd.sur_gemm_bf16(_ptr(s["dzb"]), N, 0, _ptr(s["hb"]), K, 0, _ptr(s["dw"]), K, None, N, K, M, None, 0,
                                  0, st))
        fd.check(fd.sur_bias_grad(_ptr(s["dz"]), N, M, N, _ptr(s["db"]), st))
        fd.check(fd.sur_gemm_bf16(_ptr(s["dzb"]), N, 1, _ptr(s["wb"]), K, 0, _ptr(s["dh"]), K, None, M, K, N, None, 0,
                                  0, st))
        fd.check(fd.sur_relu_bwd(_ptr(s["h"]), _ptr(s["dh"]), _ptr(s["dzp"]), _ptr(s["dzpb"]), M * K, st))
        return [s["y"], s["yb"], s["dw"], s["db"], s["dh"], s["dzp"], s["dzpb"]]
    return fd.trace_spectrum(s["x"], s["dt"], s["freqs"], t0=s["dt"], coef=s["coef"], gate=s["gate"], taper=s["taper"])


# ---- the same in 64 bits, on plain arrays ------------------------------------------------

class _Yee:
    """The 3D leapfrog (H, then E) with PEC, first-order Mur or CPML walls."""

    def __init__(self, nx, ny, nz, dx, dt, boundary, P):
        self.n, self.dx, self.dt, self.b, self.P = (nx, ny, nz), dx, dt, boundary, P
        self.eps = EPS_R / (MU0 * C0 * C0)
        self.kE, self.kH = dt / (self.eps * dx), dt / (MU0 * dx)
        S = C0 / math.sqrt(EPS_R) * dt / dx
        self.m = (S - 1.0) / (S + 1.0)
        if boundary == CPML:
            self.co = [self._coef(N) for N in self.n]

    def _coef(self, N):
        P, eta = self.P, MU0 * C0 / math.sqrt(EPS_R)
        smax = -4.0 * math.log(1e-6) / (2.0 * eta * P * self.dx)
        amax = 2.0 * math.pi * 50e6 * self.eps
        out = []
        for half in (0.0, 0.5):
            i = np.arange(N) + half
            depth = np.maximum(P - i, i - (N - P)) / P
            inside = (depth >= 0) if half == 0.0 else (depth > 0)
            x = np.where(inside, depth, 0.0)
            sg, al = smax * x ** 3, amax * (1.0 - x)
            b = np.exp(-(sg + al) * self.dt / self.eps)
            a = np.where(sg + al > 0, sg * (b - 1.0) / np.where(sg + al > 0, sg + al, 1.0), 0.0)
            keep = inside & ((i >= 1) if half == 0.0 else True)
            out += [np.where(keep, a, 0.0), np.where(keep, b, 0.0)]
        return [torch.tensor(v, device="cuda") for v in out]       # aE, bE, aH, bH by cell

    def state(self):
        nx, ny, nz = self.n
        z = lambda *s: torch.zeros(*s, dtype=torch.float64, device="cuda")
        st = [z(nz + 1, ny + 1, nx + 1) for _ in range(6)]
        if self.b == CPML:
            for ax in (2, 1, 0):       # x, y, z terms: four memory arrays each, low and high slab
                s = [nz, ny, nx]
                s[ax] = self.P + 1
                st += [z(*s) for _ in range(8)]
        return st

    def _pml(self, d, psi, ax, first, kind):
        """d (cells [first, N) of axis ax of the array axis) gains its memory in both slabs."""
        if self.b != CPML:
            return
        N, P = self.n[2 - ax], self.P
        a, b = self.co[2 - ax][2 * kind:2 * kind + 2]
        shape = [1, 1, 1]
        shape[ax] = -1
        for slab, (lo, hi) in enumerate(((0, P + 1), (N - P - 1, N))):
            lo = max(lo, first)
            v = d.narrow(ax, lo - first, hi - lo)
            m = psi[slab].narrow(ax, P + 1 - (hi - lo), hi - lo)
            m = m[tuple(slice(m.shape[t] - v.shape[t], None) for t in range(3))]   # the cells that the component updates
            m.mul_(b[lo:hi].view(shape)).add_(v * a[lo:hi].view(shape))
            v.add_(m)

    def half_h(self, st):
        nx, ny, nz = self.n
        Ex, Ey, Ez, Hx, Hy, Hz = st[:6]
        psi = lambda g, t: st[6 + 8 * g + 2 * t:8 + 8 * g + 2 * t] if self.b == CPML else None
        d1 = Ez[:nz, 1:, 1:nx] - Ez[:nz, :-1, 1:nx]
        d2 = Ey[1:, :ny, 1:nx] - Ey[:-1, :ny, 1:nx]
        self._pml(d1, psi(1, 2), 1, 0, 1)
        self._pml(d2, psi(2, 2), 0, 0, 1)
        Hx[:nz, :ny, 1:nx].sub_(d1.sub_(d2), alpha=self.kH)
        d1 = Ex[1:, 1:ny, :nx] - Ex[:-1, 1:ny, :nx]
        d2 = Ez[:nz, 1:ny, 1:] - Ez[:nz, 1:ny, :-1]
        self._pml(d1, psi(2, 3), 0, 0, 1)
        self._pml(d2, psi(0, 2), 2, 0, 1)
        Hy[:nz, 1:ny, :nx].sub_(d1.sub_(d2), alpha=self.kH)
        d1 = Ey[1:nz, :ny, 1:] - Ey[1:nz, :ny, :-1]
        d2 = Ex[1:nz, 1:, :nx] - Ex[1:nz, :-1, :nx]
        self._pml(d1, psi(0, 3), 2, 0, 1)
        self._pml(d2, psi(1, 3), 1, 0, 1)
        Hz[1:nz, :ny, :nx].sub_(d1.sub_(d2), alpha=self.kH)

    def half_e(self, st, src=None):
        nx, ny, nz = self.n
        Ex, Ey, Ez, Hx, Hy, Hz = st[:6]
        psi = lambda g, t: st[6 + 8 * g + 2 * t:8 + 8 * g + 2 * t] if self.b == CPML else None
        old = self._faces(st) if self.b == MUR else None
        d1 = Hz[1:nz, 1:ny, :nx] - Hz[1:nz, :ny - 1, :nx]
        d2 = Hy[1:nz, 1:ny, :nx] - Hy[:nz - 1, 1:ny, :nx]
        self._pml(d1, psi(1, 0), 1, 1, 0)
        self._pml(d2, psi(2, 0), 0, 1, 0)
        Ex[1:nz, 1:ny, :nx].add_(d1.sub_(d2), alpha=self.kE)
        d1 = Hx[1:nz, :ny, 1:nx] - Hx[:nz - 1, :ny, 1:nx]
        d2 = Hz[1:nz, :ny, 1:nx] - Hz[1:nz, :ny, :nx - 1]
        self._pml(d1, psi(2, 1), 0, 1, 0)
        self._pml(d2, psi(0, 0), 2, 1, 0)
        Ey[1:nz, :ny, 1:nx].add_(d1.sub_(d2), alpha=self.kE)
        d1 = Hy[:nz, 1:ny, 1:nx] - Hy[:nz, 1:ny, :nx - 1]
        d2 = Hx[:nz, 1:ny, 1:nx] - Hx[:nz, :ny - 1, 1:nx]
        self._pml(d1, psi(0, 1), 2, 1, 0)
        self._pml(d2, psi(1, 1), 1, 1, 0)
        Ez[:nz, 1:ny, 1:nx].add_(d1.sub_(d2), alpha=self.kE)
        if src is not None:
            for kk, amp, w, js, is_ in src:
                Ez[kk, js, is_].add_(w, alpha=amp)
        if old is not None:
            for f, e0, e1 in old:
                f0, f1 = self._face(st, *f)
                f0.copy_(e1 + self.m * (f1 - e0))

    def _face(self, st, ax, hi, c):
        """Tangential component c on a face (edges excluded) and next to it."""
        E, N = st[c], self.n
        s0, s1 = [None] * 3, [None] * 3
        for a in range(3):             # a: x, y, z; the array axis is 2 - a
            if a == ax:
                s0[2 - a], s1[2 - a] = (N[a], N[a] - 1) if hi else (0, 1)
            else:
                s0[2 - a] = s1[2 - a] = slice(0, N[a]) if a == c else slice(1, N[a])
        return E[tuple(s0)], E[tuple(s1)]

    def _faces(self, st):
        out = []
        for ax in range(3):
            for hi in (0, 1):
                for c in range(3):
                    if c != ax:
                        e0, e1 = self._face(st, ax, hi, c)
                        out.append(((ax, hi, c), e0.clone(), e1.clone()))
        return out

    def source(self, p, n, q=None):
        """(plane, amplitude per unit weight, weights, rows, columns) of step n's
        current; with q None per unit charge of the interpolated table."""
        nx, ny, nz = self.n
        L = p["L"]
        za, zb = p["z0"] + C0 * n * self.dt, p["z0"] + C0 * (n + 1) * self.dt
        u = C0 * (n + 0.5) * self.dt / p["bin_dz"]
        nb = len(p["q"])
        if u < 0 or u > nb - 1:
            return u, []
        if q is None:
            qbar = 1.0
        else:
            b = min(int(math.floor(u)), nb - 2)
            qbar = float(q[b]) * (1.0 - (u - b)) + float(q[b + 1]) * (u - b)
        cum = lambda z, k: 0.0 if k < math.floor(z / self.dx) else 1.0 if k > math.floor(z / self.dx) else 1.0 - (z / self.dx - math.floor(z / self.dx))
        lo, hi = (self.P, nz - self.P - 1) if self.b == CPML else (0, nz - 1)
        w = torch.tensor(p["w"], device="cuda").view(2 * L + 1, 2 * L + 1)
        js, is_ = slice(ny // 2 - L, ny // 2 + L + 1), slice(nx // 2 - L, nx // 2 + L + 1)
        out = []
        for k in range(int(math.floor(za / self.dx)) - 1, int(math.floor(zb / self.dx)) + 2):
            dC = cum(zb, k) - cum(za, k)
            if lo <= k <= hi and dC != 0.0:
                out.append((k, qbar * dC / (self.eps * self.dx ** 2), w, js, is_))
        return u, out

    def readout(self, ijk):
        nx, ny, _ = self.n
        X, Y = (ijk[:, 0] - nx // 2) * self.dx, (ijk[:, 1] - ny // 2) * self.dx
        r = np.hypot(X, Y)
        c = np.stack([X, Y], 1) / np.where(r > 0, r, 1.0)[:, None]
        i, j, k = (torch.tensor(ijk[:, a], device="cuda") for a in range(3))
        return i, j, k, torch.tensor(c, device="cuda")

    def read(self, st, rd):
        i, j, k, c = rd
        Ex, Ey, Ez = st[:3]
        ex, ey, ez = 0.5 * (Ex[k, j, i - 1] + Ex[k, j, i]), 0.5 * (Ey[k, j - 1, i] + Ey[k, j, i]), 0.5 * (Ez[k - 1, j, i] + Ez[k, j, i])
        return torch.stack([ez, c[:, 0] * ex + c[:, 1] * ey], 1)

    def forward(self, p, q, steps):
        st, rd = self.state(), self.readout(p["ijk"])
        tr = torch.zeros(len(p["ijk"]), steps, 2, dtype=torch.float64, device="cuda")
        for n in range(steps):
            self.half_h(st)
            self.half_e(st, self.source(p, n, q)[1])
            tr[:, n] = self.read(st, rd)
        return tr, st

    def gradient(self, p, g, steps):
        """d(sum g trace)/dq: the transpose of every step by autograd, last to first."""
        zero, rd = self.state(), self.readout(p["ijk"])
        i, j, k, c = rd
        mu = [torch.zeros_like(x) for x in zero]
        grad = torch.zeros(len(p["q"]), dtype=torch.float64)
        for n in reversed(range(steps)):
            gz, gx, gy = 0.5 * g[:, n, 0], 0.5 * c[:, 0] * g[:, n, 1], 0.5 * c[:, 1] * g[:, n, 1]
            for comp, at, v in ((0, (k, j, i - 1), gx), (0, (k, j, i), gx), (1, (k, j - 1, i), gy), (1, (k, j, i), gy),
                                (2, (k - 1, j, i), gz), (2, (k, j, i), gz)):
                mu[comp].index_put_(at, v, accumulate=True)
            u, src = self.source(p, n)
            d = sum(float((mu[2][kk, js, is_] * w).sum()) * amp for kk, amp, w, js, is_ in src)
            if src:
                b = min(int(math.floor(u)), len(p["q"]) - 2)
                grad[b] += (1.0 - (u - b)) * d
                grad[b + 1] += (u - b) * d
            if n > 0:
                with torch.enable_grad():
                    leaf = [x.requires_grad_(True) for x in zero]
                    st = [x.clone() for x in leaf]
                    self.half_h(st)
                    self.half_e(st)
                    mu = list(torch.autograd.grad(st, leaf, mu))
                zero = [x.detach() for x in zero]
        return grad


def _exact_cyl(case, seed):
    p = _cyl_inputs(case, seed)
    nr, nz, d, dt = case["nr"], case["nz"], p["d"], p["dt"]
    eps = EPS_R / (MU0 * C0 * C0)
    kE, kH = dt / (eps * d), dt / (MU0 * d)
    S = C0 / math.sqrt(EPS_R) * dt / d
    m = (S - 1.0) / (S + 1.0) if case["boundary"] == MUR else None
    z = lambda *s: torch.zeros(*s, dtype=torch.float64, device="cuda")
    Er, Ez, Hp = z(nr, nz + 1), z(nr + 1, nz), z(nr, nz)
    i = torch.arange(1, nr, dtype=torch.float64, device="cuda")[:, None]
    cA, cB = kE * (i + 0.5) / i, kE * (i - 0.5) / i
    nw = min(len(p["w"]), nr)
    ring = torch.arange(nw, dtype=torch.float64)
    area = 2.0 * math.pi * ring * d * d
    area[0] = math.pi * d * d / 4.0
    wr = (torch.tensor(p["w"][:nw]) / (eps * area)).cuda()
    ii, jj = (torch.tensor(p["ij"][:, a], device="cuda") for a in (0, 1))
    tr = z(case["probes"], case["steps"] + 800, 2)
    nb = len(p["q"])
    cum = lambda x, j: (1.0 - (x - math.floor(x)) if j >= math.floor(x) else 0.0) + (x - math.floor(x) if j >= math.floor(x) + 1 else 0.0)
    for n in range(case["steps"]):
        dH = Er[:, 1:] - Er[:, :-1]
        dH.sub_(Ez[1:] - Ez[:-1])
        Hp.sub_(dH, alpha=kH)
        if m is not None:
            lo, hi = (Er[:, 0].clone(), Er[:, 1].clone()), (Er[:, nz].clone(), Er[:, nz - 1].clone())
            wall = Ez[nr].clone(), Ez[nr - 1].clone()
        Er[:, 1:nz].sub_(Hp[:, 1:] - Hp[:, :-1], alpha=kE)
        Ez[1:nr].addcmul_(Hp[1:], cA.expand(-1, nz)).addcmul_(Hp[:-1], cB.expand(-1, nz), value=-1.0)
        Ez[0].add_(Hp[0], alpha=4.0 * kE)
        xa, xb = (p["z0"] + C0 * n * dt) / d, (p["z0"] + C0 * (n + 1) * dt) / d
        u = C0 * (n + 0.5) * dt / p["bin_dz"]
        if 0 <= u <= nb - 1:
            b = min(int(math.floor(u)), nb - 2)
            qb = p["q"][b] * (1.0 - (u - b)) + p["q"][b + 1] * (u - b)
            for j in range(int(math.floor(xa)) - 1, int(math.floor(xb)) + 2):
                dC = cum(xb, j) - cum(xa, j)
                if dC != 0.0 and 0 <= j < nz:
                    Ez[:nw, j].add_(wr, alpha=qb * dC)
        if m is not None:
            Er[:, 0] = lo[1] + m * (Er[:, 1] - lo[0])
            Er[:, nz] = hi[1] + m * (Er[:, nz - 1] - hi[0])
            Ez[nr] = wall[1] + m * (Ez[nr - 1] - wall[0])
        ez = 0.5 * (Ez[ii, jj - 1] + Ez[ii, jj])
        er = torch.where(ii > 0, 0.5 * (Er[(ii - 1).clamp_min(0), jj] + Er[ii, jj]), torch.zeros_like(ez))
        tr[:, n] = torch.stack([ez, er], 1)
    return [tr, Er, Ez, Hp]


def _lattice_taps(case, ant, k):
    """Table rows and sample range of bin k's responses: (rows [n], first tau, first t, length)."""
    T, S = case["T"], case["S"]
    D = case["m_hi"] - case["m_lo"] + case["K"]
    row = ant[:, 0].long() * D + (ant[:, 1].long() - k + case["K"] - 1 - case["m_lo"])
    off = S * k - S                    # t = tau + off
    t0 = max(0, off)
    return row, t0 - off, t0, T - max(t0, t0 - off)


def _exact_lattice(case, seed):
    p = _lattice_inputs(case, seed)
    K, T = case["K"], case["T"]
    G = p["G"].double().reshape(-1, T)
    q = p["q"].double()
    s = q.abs().amax(1)
    qn = q / s[:, None]
    if case["kind"] == "lattice_serve":
        P, A = q.shape[0], p["ant"].shape[0]
        W = torch.zeros(A, K, T, dtype=torch.float64, device="cuda")
        for k in range(K):
            row, tau, t, n = _lattice_taps(case, p["ant"], k)
            if n > 0:
                W[:, k, t:t + n] = G[row, tau:tau + n]
        y = torch.empty(A, P, T, dtype=torch.float64, device="cuda")
        for a in range(A):
            torch.matmul(qn, W[a], out=y[a])
        return y.mul_((s * p["c_out"])[None, :, None])
    B = q.shape[0]
    y = torch.zeros(B, T, dtype=torch.float64, device="cuda")
    for k in range(K):
        row, tau, t, n = _lattice_taps(case, p["ant"], k)
        if n > 0:
            y[:, t:t + n] += qn[:, k:k + 1] * G[row, tau:tau + n]
    target, st = p["trace"].double(), None
    if case["relative"]:
        st = target.abs().amax(1, keepdim=True)
        y, target = y * (p["c_out"] * s[:, None] / st), target / st
    else:
        target = target / (p["c_out"] * s[:, None])
    loss = ((y - target) ** 2).mean()
    dy = 2.0 * (y - target) / (B * T)
    if case["relative"]:
        dy = dy * (p["c_out"] * s[:, None] / st)
    dG = torch.zeros_like(G)
    for k in range(K):
        row, tau, t, n = _lattice_taps(case, p["ant"], k)
        if n > 0:
            dG[:, tau:tau + n].index_add_(0, row, qn[:, k:k + 1] * dy[:, t:t + n])
    t, b1, b2 = 5001, 0.9, 0.999
    m = b1 * p["m"].double() + (1 - b1) * dG.view_as(p["m"])
    v = b2 * p["v"].double() + (1 - b2) * dG.view_as(p["v"]) ** 2
    G = G.view_as(m) - 1e-3 * (m / (1 - b1 ** t)) / (torch.sqrt(v / (1 - b2 ** t)) + 1e-8)
    return [loss.view(1), G, m, v]


def exact(case, seed):
    k = case["kind"]
    if k == "fdtd":
        p = _fdtd_inputs(case, seed)
        y = _Yee(case["nx"], case["ny"], case["nz"], case["dx"], p["dt"], case["boundary"], case["npml"])
        tr, st = y.forward(p, p["q"], case["steps"])
        return [tr, torch.stack(st[:3]), torch.stack(st[3:6])]
    if k == "adjoint":
        p = _adjoint_inputs(case, seed)
        y = _Yee(case["nx"], case["ny"], case["nz"], 0.02, p["dt"], case["boundary"], case["npml"])
        q = p["q"].astype(np.float64)
        tr = y.forward(p, q, case["steps"])[0]
        res = y.forward(p, q - p["q_true"].astype(np.float64), case["steps"])[0]
        return [tr, y.gradient(p, res, case["steps"])]
    if k == "batch":
        traces, fields = [], [[] for _ in range(6)]
        for p in _batch_inputs(case, seed):
            y = _Yee(p["nx"], p["ny"], p["nz"], 0.02, p["dt"], MUR, 0)
            tr, st = y.forward(p, p["q"], case["steps"])
            traces.append(torch.nn.functional.pad(tr, (0, 0, 0, 1000 - case["steps"])))
            for c in range(6):
                fields[c].append(st[c].reshape(-1))
        fields = [torch.cat(f) for f in fields]
        return [torch.stack(traces), torch.stack(fields[:3]), torch.stack(fields[3:])]
    if k == "cyl":
        return _exact_cyl(case, seed)
    if k in ("lattice_train", "lattice_serve"):
        return _exact_lattice(case, seed)
    if k == "mlp_layer":
        p = _mlp_inputs(case, seed)
        h, w, dz = p["hb"].double(), p["wb"].double(), p["dzb"].double()
        y = h @ w.T + p["bias"].double()
        y = y.clamp_min(0.0) if case["relu"] else y
        dh = dz @ w
        dzp = torch.where(p["h"] > 0, dh, torch.zeros_like(dh))
        return [y, y, dz.T @ h, p["dz"].double().sum(0), dh, dzp, dzp]
    p = _spectrum_inputs(case, seed)
    n, T = case["traces"], case["samples"]
    x = (p["x"].double() * torch.tensor(p["coef"], device="cuda")[:, None, :]).sum(2)
    gate = p["gate"] if p["gate"] is not None else np.tile(np.array([[0, T]]), (n, 1))
    first, count = (torch.tensor(gate[:, a].astype(np.int64), device="cuda")[:, None] for a in (0, 1))
    at = torch.arange(T, device="cuda")[None, :] - first
    u = at.double() / (count - 1).clamp_min(1).double()
    win = ((at >= 0) & (at < count)).double()
    if case["taper"] > 0:
        e = torch.minimum(u, 1.0 - u).clamp_min(0.0)
        ramp = 0.5 * (1.0 - torch.cos(2.0 * math.pi * e / case["taper"]))
        win = win * torch.where((e < 0.5 * case["taper"]) & (count > 1), ramp, torch.ones_like(ramp))
    x = x * win
    f = torch.tensor(p["freqs"], device="cuda")
    t = (torch.arange(T, device="cuda").double() + 1.0) * p["dt"]
    out = torch.zeros(n, len(p["freqs"]), dtype=torch.complex128, device="cuda")
    for lo in range(0, T, 4096):
        ph = 2.0 * math.pi * torch.remainder(t[lo:lo + 4096, None] * f[None, :], 1.0)
        out += torch.complex(x[:, lo:lo + 4096] @ torch.cos(ph), x[:, lo:lo + 4096] @ torch.sin(ph))
    return out * p["dt"]
