"""Performance cases of the library: the work its users have it do, through the Python binding.

Each case is one call (or one forward and backward pass) of a public entry point on a lattice
that the caller keeps, with the caller's start vectors and work buffer: KPM moments of the three
models in the three precisions, the batched KPM of many lattices, a Chebyshev filter, the
spectral function, graphene wave-packet propagation and its gradient, and one fused Chebyshev
step of a caller's own iteration on a small lattice.  `exact` computes the same results in
64 bits with plain torch operations, from the model equations.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1708_09689_gb300 as pv

PREC = {"c64": pv.C64, "c128": pv.C128, "q64": pv.Q64}
VEC = {"c64": torch.complex64, "c128": torch.complex128, "q64": torch.complex128}
CBYTES = {"c64": 8, "c128": 16, "q64": 16}
L2_BYTES = 129e6


def _dev() -> str:
    return "cuda" if torch.cuda.is_available() else "cpu"


# ------------------------------------------------------------------------------- the cases
def listed() -> list[dict]:
    return [
        # one fused step (H x, shift, scale, dot products) of a caller's own Krylov or Chebyshev
        # iteration on a small sample: launch latency and host time
        {"name": "step_small_c128", "kind": "step", "nx": 24, "ny": 20, "nz": 18, "px": 1, "py": 1, "pz": 0,
         "R": 4, "prec": "c128", "W": 1.0},
        # moments of one random vector on the 16^3 cube of the accuracy runs: a chain of 128 sweeps
        # of a few microseconds each
        {"name": "kpm_cube_c128", "kind": "kpm", "model": "ti", "nx": 16, "ny": 16, "nz": 16, "px": 1, "py": 1,
         "pz": 1, "R": 1, "prec": "c128", "M": 256, "W": 1.0, "tuned": 0},
        # the headline run: density of states of a disordered slab, complex64 blocks of 8 vectors, in
        # the launch shape a tuned program keeps
        {"name": "kpm_slab_c64_tuned", "kind": "kpm", "model": "ti", "nx": 256, "ny": 256, "nz": 64, "px": 1,
         "py": 1, "pz": 0, "R": 8, "prec": "c64", "M": 64, "W": 2.0, "tuned": 1},
        # a reference run in full double precision on a quarter of that slab
        {"name": "kpm_cuboid_c128", "kind": "kpm", "model": "ti", "nx": 128, "ny": 128, "nz": 64, "px": 1, "py": 1,
         "pz": 0, "R": 8, "prec": "c128", "M": 32, "W": 2.0, "tuned": 0},
        # a sample whose lengths are no round numbers, open on all sides, with default settings
        {"name": "kpm_ragged_c64", "kind": "kpm", "model": "ti", "nx": 101, "ny": 87, "nz": 53, "px": 0, "py": 0,
         "pz": 0, "R": 4, "prec": "c64", "M": 128, "W": 1.5, "tuned": 0},
        # fp64-accurate moments on 64-bit fixed-point vectors
        {"name": "kpm_cuboid_q64", "kind": "kpm", "model": "ti", "nx": 128, "ny": 128, "nz": 64, "px": 1, "py": 1,
         "pz": 0, "R": 8, "prec": "q64", "M": 64, "W": 2.0, "tuned": 0},
        # the Weyl-semimetal cuboid of the dispersion figure, default settings
        {"name": "kpm_weyl_c64", "kind": "kpm", "model": "wsm", "nx": 256, "ny": 32, "nz": 32, "px": 1, "py": 1,
         "pz": 0, "R": 16, "prec": "c64", "M": 256, "W": 1.0, "tuned": 0},
        # a wave packet on the quantum-dot array, 2^25 sites: two time steps, complex64 recurrence with
        # the state in double precision
        {"name": "propagate_qd_c64", "kind": "propagate", "nx": 4096, "ny": 2048, "px": 0, "py": 0, "R": 1,
         "prec": "c64", "steps": 2, "dots": 8, "radius": 40.0},
        # gate-potential gradient: forward with checkpoints and the adjoint, complex128
        {"name": "gradient_qd_c128", "kind": "gradient", "nx": 512, "ny": 256, "px": 0, "py": 0, "steps": 10,
         "every": 5, "dots": 4, "radius": 15.0},
        # the filter of a filter diagonalization on its thin slab
        {"name": "filter_slab_c64", "kind": "filter", "nx": 240, "ny": 240, "nz": 6, "px": 1, "py": 1, "pz": 0,
         "R": 32, "prec": "c64", "K": 100, "W": 1.0},
        # A(k, E) of eight k-points on a thin cuboid, the whole call
        {"name": "spectral_c64", "kind": "spectral", "nx": 256, "ny": 64, "nz": 8, "px": 1, "py": 1, "pz": 1,
         "nk": 8, "M": 256, "NE": 1024, "prec": "c64", "W": 0.0},
        # disorder average: sixteen cubes of uneven size in one call
        {"name": "batched_c64", "kind": "batched", "n": 16, "Lmin": 24, "Lmax": 64, "R": 16, "M": 64,
         "prec": "c64", "W": 5.0},
    ]


def _log(rng, lo, hi) -> int:
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng) -> dict:
    kind = rng.choice(["kpm", "kpm", "kpm", "kpm", "step", "propagate", "gradient", "filter", "spectral", "batched"])
    per = [rng.randint(0, 1) for _ in range(3)]
    if kind == "kpm":
        model = rng.choice(["ti", "ti", "wsm"])
        prec = rng.choice(["c64", "c64", "c128"] + (["q64"] if model == "ti" else []))
        R = rng.choice([1, 2, 4, 8, 16, 32])
        while True:
            nx, ny, nz = _log(rng, 12, 300), _log(rng, 12, 300), _log(rng, 4, 100)
            if nx * ny * nz * R <= (1 << 25 if prec == "c64" else 1 << 23):
                break
        if model == "wsm":
            nx += nx & 1
        return {"kind": kind, "model": model, "nx": nx, "ny": ny, "nz": nz, "px": per[0], "py": per[1],
                "pz": per[2], "R": R, "prec": prec, "M": _log(rng, 9, 32 if prec == "c128" else 64),
                "W": rng.choice([0.0, 1.0, 2.5]), "tuned": 0}
    if kind == "step":
        return {"kind": kind, "nx": _log(rng, 8, 200), "ny": _log(rng, 8, 100), "nz": _log(rng, 4, 30),
                "px": per[0], "py": per[1], "pz": per[2], "R": rng.choice([1, 2, 4, 8]),
                "prec": rng.choice(["c64", "c128"]), "W": rng.choice([0.0, 2.0])}
    if kind == "propagate":
        return {"kind": kind, "nx": _log(rng, 60, 2000), "ny": _log(rng, 60, 1500), "px": per[0], "py": per[1],
                "R": rng.choice([1, 1, 2]), "prec": rng.choice(["c64", "c128"]), "steps": rng.randint(1, 2),
                "dots": rng.randint(2, 8), "radius": float(rng.randint(5, 20))}
    if kind == "gradient":
        return {"kind": kind, "nx": _log(rng, 40, 500), "ny": _log(rng, 40, 300), "px": per[0], "py": per[1],
                "steps": rng.randint(3, 8), "every": rng.randint(2, 5), "dots": rng.randint(2, 4),
                "radius": float(rng.randint(5, 15))}
    if kind == "filter":
        return {"kind": kind, "nx": _log(rng, 40, 240), "ny": _log(rng, 40, 240), "nz": _log(rng, 4, 12),
                "px": per[0], "py": per[1], "pz": per[2], "R": rng.choice([4, 8, 16]),
                "prec": "c64", "K": _log(rng, 5, 100), "W": rng.choice([0.0, 1.0])}
    if kind == "spectral":
        prec = rng.choice(["c64", "c64", "c128"])
        while True:
            nx, ny, nz, nk, M = (_log(rng, 32, 256), _log(rng, 16, 64), _log(rng, 4, 16),
                                 rng.choice([1, 2, 4, 8]), _log(rng, 64, 256))
            if nx * ny * nz * 2 * nk * M <= (5e8 if prec == "c64" else 1e8):
                break
        return {"kind": kind, "nx": nx, "ny": ny, "nz": nz, "px": 1, "py": 1, "pz": per[2], "nk": nk, "M": M,
                "NE": _log(rng, 100, 2000), "prec": prec, "W": rng.choice([0.0, 1.0])}
    return {"kind": kind, "n": rng.randint(3, 16), "Lmin": rng.randint(8, 24), "Lmax": rng.randint(25, 56),
            "R": rng.choice([4, 8, 16]), "M": _log(rng, 16, 64), "prec": "c64", "W": rng.choice([2.0, 5.0])}


# ------------------------------------------------------------------------------- inputs
def _gen(seed: int, stream: int) -> torch.Generator:
    g = torch.Generator(device=_dev())
    g.manual_seed(1000003 * int(seed) + stream)
    return g


def _dims(case):
    return case["nx"], case["ny"], case["nz"]


def _periodic(case):
    return case["px"], case["py"], case["pz"]


def _orbitals(case) -> int:
    return 2 if case.get("model") == "wsm" else 4


def _box(n: int, W: float, seed: int, stream: int = 1) -> torch.Tensor:
    """On-site box disorder in [-W/2, W/2)."""
    return W * (torch.rand(n, generator=_gen(seed, stream), device=_dev(), dtype=torch.float64) - 0.5)


def _phases(D: int, R: int, dtype, seed: int, stream: int = 2) -> torch.Tensor:
    """Random-phase vectors of unit norm, the start vectors of stochastic traces."""
    u = torch.rand((D, R), generator=_gen(seed, stream), device=_dev(), dtype=torch.float64)
    return torch.polar(torch.full_like(u, 1.0 / math.sqrt(D)), 2.0 * math.pi * u).to(dtype)


def _scaling(case) -> tuple[float, float]:
    """(a, b) from the row sums of the model: every eigenvalue of (H - b)/a lies inside (-1, 1)."""
    if case["kind"] in ("propagate", "gradient"):
        return 3.0 + 0.06, 0.05  # 3 t, dots of height 0.1
    rows = 6.0 if case.get("model") == "wsm" else 8.0  # c0 + 4 and |m| + 6 t
    return 1.002 * (rows + 0.5 * case["W"]), 0.0


def _positions(nx: int, ny: int):
    """Physical coordinates (X, Y) of the sites of nx x ny four-site cells, shape (ny, nx, 4)."""
    s3 = math.sqrt(3.0)
    d = {"device": _dev(), "dtype": torch.float64}
    x = torch.arange(nx, **d)[None, :, None]
    y = torch.arange(ny, **d)[:, None, None]
    X = 3.0 * y + torch.tensor([0.0, 0.5, 1.5, 2.0], **d) + 0.0 * x
    Y = s3 * x + torch.tensor([s3 / 2, 0.0, 0.0, s3 / 2], **d) + 0.0 * y
    return X, Y


def _dot_potential(case) -> torch.Tensor:
    """A square array of gate-defined dots, height 0.1, smooth edges of width 5, spacing 4 radii."""
    X, Y = _positions(case["nx"], case["ny"])
    K, Rd = case["dots"], case["radius"]
    d2 = torch.zeros_like(X)
    for Q, size in ((X, 3.0 * case["ny"]), (Y, math.sqrt(3.0) * case["nx"])):
        q0 = 0.5 * size - 2.0 * Rd * (K - 1)
        k = torch.clamp(torch.round((Q - q0) / (4.0 * Rd)), 0, K - 1)
        d2 += (Q - (q0 + 4.0 * Rd * k)) ** 2
    return (0.05 * (1.0 + torch.tanh((Rd - torch.sqrt(d2)) / 5.0))).reshape(-1)


def _packets(case, seed: int) -> torch.Tensor:
    """R Gaussian wave packets, each with its own centre and wave vector near the Dirac point."""
    X, Y = _positions(case["nx"], case["ny"])
    R = case.get("R", 1)
    h = torch.rand((R, 4), generator=_gen(seed, 3), device=_dev(), dtype=torch.float64)
    out = torch.empty((X.numel(), R), dtype=torch.complex128, device=_dev())
    lx, ly = 3.0 * case["ny"], math.sqrt(3.0) * case["nx"]
    width = min(50.0, 0.1 * min(lx, ly) + 1.0)
    for r in range(R):
        cx, cy = (0.25 + 0.5 * h[r, 0]) * lx, (0.25 + 0.5 * h[r, 1]) * ly
        kx, ky = 0.1 * h[r, 2], 4.0 * math.pi / (3.0 * math.sqrt(3.0)) + 0.1 * (h[r, 3] - 0.5)
        env = torch.exp(-((X - cx) ** 2 + (Y - cy) ** 2) / (4.0 * width * width))
        psi = torch.polar(env, kx * X + ky * Y).reshape(-1)
        out[:, r] = psi / torch.linalg.vector_norm(psi)
    return out if R > 1 else out[:, 0].contiguous()


def _filter_weights(K: int) -> list[float]:
    """Chebyshev coefficients of a window around the band centre with Jackson damping."""
    lo, hi = math.acos(0.04), math.acos(-0.04)
    g = []
    for k in range(K):
        c = (hi - lo) / math.pi if k == 0 else 2.0 * (math.sin(k * hi) - math.sin(k * lo)) / (k * math.pi)
        q = math.pi / (K + 1)
        g.append(c * ((K - k + 1) * math.cos(q * k) + math.sin(q * k) / math.tan(q)) / (K + 1))
    return g


def _k_points(case, seed: int):
    j0 = int(torch.randint(0, 1000, (1,), generator=_gen(seed, 4), device=_dev()))
    return [(2.0 * math.pi * ((j0 + 3 * q) % case["nx"]) / case["nx"],
             2.0 * math.pi * ((j0 // 7 + q) % case["ny"]) / case["ny"], 0.0) for q in range(case["nk"])]


def _energies(case) -> torch.Tensor:
    a, b = _scaling(case)
    return torch.linspace(b - 0.95 * a, b + 0.95 * a, case["NE"], dtype=torch.float64, device=_dev())


def _cubes(case, seed: int):
    """(L, V) of every cube of a batch: lengths in steps over [Lmin, Lmax], each with its own disorder."""
    n = case["n"]
    out = []
    for i in range(n):
        L = case["Lmin"] + (case["Lmax"] - case["Lmin"]) * ((5 * i) % n) // max(n - 1, 1)
        out.append((L, _box(L ** 3, case["W"], seed, 100 + i)))
    return out


def prepare(case, seed):
    kind = case["kind"]
    a, b = (None, None) if kind == "batched" else _scaling(case)
    s = {"case": case, "a": a, "b": b}
    if kind in ("kpm", "step", "filter", "spectral"):
        V = _box(math.prod(_dims(case)), case["W"], seed) if case["W"] else None
        make = pv.Lattice.wsm if case.get("model") == "wsm" else pv.Lattice.ti
        lat = s["lat"] = make(_dims(case), _periodic(case), V=V)
        prec = s["prec"] = PREC[case["prec"]]
    if kind == "kpm":
        R, M = case["R"], case["M"]
        s["r0"] = _phases(lat.D, R, VEC[case["prec"]], seed)
        if case["tuned"]:
            lat.set_tuning(R, prec, kernel=7)
        s["work"] = pv.work_buffer(lat.work_bytes(pv.OP_KPM, R, prec, M))
        s["mu"] = torch.empty((R, M), dtype=torch.float64, device=_dev())
    elif kind == "step":
        s["x"] = _phases(lat.D, case["R"], VEC[case["prec"]], seed)
        s["y"] = torch.empty_like(s["x"])
        s["work"] = pv.work_buffer(lat.work_bytes(pv.OP_CHEB_STEP, case["R"], prec))
    elif kind == "filter":
        s["x"] = _phases(lat.D, case["R"], torch.complex128, seed)
        s["g"] = _filter_weights(case["K"])
        s["work"] = pv.work_buffer(lat.work_bytes(pv.OP_SERIES, case["R"], prec, case["K"]))
    elif kind == "spectral":
        s["ks"] = _k_points(case, seed)
        s["E"] = _energies(case)
    elif kind in ("propagate", "gradient"):
        V = s["V"] = _dot_potential(case)
        s["psi"] = _packets(case, seed)
        lat = s["lat"] = pv.Lattice.graphene((case["nx"], case["ny"]), (case["px"], case["py"]), V=V)
        if kind == "propagate":
            prec = s["prec"] = PREC[case["prec"]]
            K = len(pv.propagation_coeffs(a * 1.0))
            s["work"] = pv.work_buffer(lat.work_bytes(pv.OP_SERIES, case["R"], prec, K))
        else:
            s["V"].requires_grad_(True)
            s["psi"].requires_grad_(True)
            s["mask"] = _detector(case)
    else:
        cubes = _cubes(case, seed)
        s["lats"] = [pv.Lattice.ti((L, L, L), (1, 1, 1), V=V) for L, V in cubes]
        s["ab"] = _batch_scaling(case)
        s["seeds"] = [int(seed) * 1000 + i for i in range(case["n"])]
        s["prec"] = PREC[case["prec"]]
        s["work"] = pv.work_buffer(pv.batched_work_bytes(s["lats"], case["R"], s["prec"], case["M"]))
    return s


def _detector(case) -> torch.Tensor:
    """Sites of the detector behind the array, the last quarter along physical X."""
    X, _ = _positions(case["nx"], case["ny"])
    return (X.reshape(-1) > 0.75 * 3.0 * case["ny"]).to(torch.float64)


def _batch_scaling(case):
    a = 1.002 * (8.0 + 0.5 * case["W"])
    return [a] * case["n"], [0.0] * case["n"]


def run(state):
    s, case = state, state["case"]
    kind = case["kind"]
    if kind == "kpm":
        return pv.kpm_moments(s["lat"], case["M"], s["a"], s["b"], prec=s["prec"], r0=s["r0"], work=s["work"],
                              mu=s["mu"])
    if kind == "step":
        R = case["R"]
        d = pv.cheb_step(s["lat"], s["x"], s["y"], [1.0 / s["a"]] * R, [s["b"]] * R, dots=7, work=s["work"])
        return {"y": s["y"], "dots": d}
    if kind == "filter":
        return pv.cheb_filter(s["lat"], s["x"], s["g"], s["a"], s["b"], prec=s["prec"], work=s["work"])
    if kind == "spectral":
        return pv.spectral_function(s["lat"], s["ks"], case["M"], s["a"], s["b"], s["E"], prec=s["prec"])
    if kind == "propagate":
        return pv.cheb_propagate(s["lat"], s["psi"].clone(), 1.0, case["steps"], s["a"], s["b"], prec=s["prec"],
                                 work=s["work"])
    if kind == "gradient":
        psi = pv.propagate_with_grad(s["V"], s["psi"], s["lat"], 1.0, case["steps"], s["a"], s["b"],
                                     every=case["every"])
        loss = (psi.abs() ** 2 * s["mask"]).sum()
        gV, gpsi = torch.autograd.grad(loss, (s["V"], s["psi"]))
        return {"loss": loss.detach(), "psi": psi.detach(), "gV": gV, "gpsi": gpsi}
    return pv.kpm_moments_batched(s["lats"], case["M"], *s["ab"], R=case["R"], prec=s["prec"], seeds=s["seeds"],
                                  work=s["work"])


# ------------------------------------------------------------------------------- least work
# Operations of one site and vector: the TI hopping by its rank-2 bond matrices (6 x 4 additions to
# project a neighbour, 2 x 5 x 4 to sum), the update (8 x 5) and two dot products (2 x 16); the Weyl
# semimetal half of that.
TI_FLOPS = 24.0 + 40.0 + 40.0 + 32.0
WSM_FLOPS = 0.5 * TI_FLOPS


def _sweep_work(sites, R, comp, cb, vb, sweeps, extra=0.0, flops=0.0):
    """Bytes and operations of a chain of fused sweeps on `sites` sites of `comp` components: per
    sweep two vector blocks read and one written and the potential read (vb bytes a site), or, for
    blocks that stay in the L2 cache, the first read and the last write alone."""
    block = float(sites) * comp * R * cb
    per = 3.0 * block + float(sites) * vb
    if 2.0 * block + sites * vb <= 0.5 * L2_BYTES:
        bytes_ = per + extra
    else:
        bytes_ = sweeps * per + extra
    return {"bytes": bytes_, "flops": float(sites) * R * sweeps * flops}


def work(case):
    kind = case["kind"]
    if kind == "step":
        n, R, cb = math.prod(_dims(case)), case["R"], CBYTES[case["prec"]]
        return {"bytes": 2.0 * n * 4 * R * cb + 8.0 * n * (case["W"] > 0), "flops": TI_FLOPS * n * R}
    if kind in ("kpm", "spectral"):
        sites, sweeps = math.prod(_dims(case)), (case["M"] + 1) // 2
        R = case["R"] if kind == "kpm" else 4 * case["nk"]
        cb = CBYTES[case["prec"]]
        vb = (4.0 if case["prec"] == "c64" else 8.0 if case["prec"] == "c128" else 16.0) * (case["W"] > 0)
        return _sweep_work(sites, R, _orbitals(case), cb, vb, sweeps,
                           flops=TI_FLOPS if case.get("model") != "wsm" else WSM_FLOPS)
    if kind == "filter":
        sites, K = math.prod(_dims(case)), case["K"]
        acc = 2.0 * sites * 4 * case["R"] * 16 * (K / 3.0 + 1)
        return _sweep_work(sites, case["R"], 4, 8, 4.0 * (case["W"] > 0), K - 1, extra=acc, flops=TI_FLOPS)
    if kind == "propagate":
        sites, K = 4 * case["nx"] * case["ny"], 20
        acc = 2.0 * sites * case["R"] * 16 * (K / 3.0 + 1) * case["steps"]
        cb = CBYTES[case["prec"]]
        return _sweep_work(sites, case["R"], 1, cb, cb / 2.0, (K - 1) * case["steps"], extra=acc, flops=22.0)
    if kind == "gradient":
        # forward, recomputed states, and per adjoint step the forward and the reverse recurrence
        sites, K = 4 * case["nx"] * case["ny"], 20
        seg = case["steps"] - (case["steps"] + case["every"] - 1) // case["every"]
        sweeps = (K - 1) * (case["steps"] + seg + 2 * case["steps"])
        return _sweep_work(sites, 1, 1, 16, 8.0, sweeps, flops=26.0)
    sites = sum(L ** 3 for L in _cube_lengths(case))
    return _sweep_work(sites, case["R"], 4, 8, 4.0, (case["M"] + 1) // 2, flops=TI_FLOPS)


def _cube_lengths(case):
    n = case["n"]
    return [case["Lmin"] + (case["Lmax"] - case["Lmin"]) * ((5 * i) % n) // max(n - 1, 1) for i in range(n)]


# ------------------------------------------------------------------------------- in 64 bits
def _shift(x, axis: int, step: int, periodic: bool):
    """x at the neighbour one site further (step +1) or back (-1) along a tensor axis; zero past an open edge."""
    y = torch.roll(x, -step, dims=axis)
    if not periodic:
        y.select(axis, x.shape[axis] - 1 if step > 0 else 0).zero_()
    return y


def _ti_apply(x, V, per, m=2.0, t=1.0):
    """H x of the cubic topological insulator; x (Lz, Ly, Lx, 4, R), V (Lz, Ly, Lx) or None."""
    sign = torch.tensor([1.0, -1.0, 1.0, -1.0], dtype=torch.float64, device=x.device)[:, None]
    diag = m * sign
    y = diag * x if V is None else (V[..., None, None] + diag) * x
    for axis, ax in ((0, 2), (1, 1), (2, 0)):  # lattice axis x, y, z is tensor axis 2, 1, 0
        back, fwd = _shift(x, ax, -1, per[axis]), _shift(x, ax, 1, per[axis])
        y -= 0.5 * t * sign * (back + fwd)
        d = back - fwd
        d0, d1, d2, d3 = (d[..., o, :] for o in range(4))
        turned = ((d3, d2, -d1, -d0), (-1j * d3, -1j * d2, -1j * d1, -1j * d0), (d1, -d0, d3, -d2))[axis]
        y -= 0.5 * t * torch.stack(turned, dim=-2)
    return y


def _wsm_apply(x, V, per, k0=math.pi / 2):
    """H x of the two-band Weyl semimetal; x (Lz, Ly, Lx, 2, R)."""
    c0 = 2.0 + math.cos(k0)
    s = lambda ax, step: _shift(x, ax, step, per[2 - ax])  # noqa: E731
    xs, zm, zp = 0.5 * (s(2, -1) + s(2, 1)), s(0, -1), s(0, 1)
    ym, yp = s(1, -1), s(1, 1)
    zs, dz = 0.5 * (zm + zp), 0.5j * (zm - zp)
    a = -c0 * x[..., 1, :] + xs[..., 1, :] + ym[..., 1, :] + zs[..., 1, :] + dz[..., 0, :]
    b = -c0 * x[..., 0, :] + xs[..., 0, :] + yp[..., 0, :] + zs[..., 0, :] - dz[..., 1, :]
    y = torch.stack((a, b), dim=-2)
    return y if V is None else y + V[..., None, None] * x


def _graphene_apply(x, V, per, t=1.0):
    """H x of graphene in four-site cells; x (Ny, Nx, 4, R), V (Ny, Nx, 4)."""
    c = [x[..., o, :] for o in range(4)]
    xp = lambda o: _shift(c[o], 1, 1, per[0])   # noqa: E731
    xm = lambda o: _shift(c[o], 1, -1, per[0])  # noqa: E731
    n = (c[1] + xp(1) + _shift(c[3], 0, -1, per[1]), c[0] + c[2] + xm(0),
         c[1] + c[3] + xm(3), c[2] + xp(2) + _shift(c[0], 0, 1, per[1]))
    return V[..., None] * x - t * torch.stack(n, dim=-2)


def _operator(case, V):
    """H~ = (H - b)/a on flat (D, R) blocks."""
    a, b = _scaling(case)
    if case["kind"] in ("propagate", "gradient"):
        shape, per, f = (case["ny"], case["nx"]), (case["px"], case["py"]), _graphene_apply
        Vs = V.reshape(shape + (4,))
        comp = 4
    else:
        nx, ny, nz = _dims(case)
        shape, per, comp = (nz, ny, nx), _periodic(case), _orbitals(case)
        f = _wsm_apply if comp == 2 else _ti_apply
        Vs = None if V is None else V.reshape(shape)

    def apply(x):
        R = x.shape[1]
        return ((f(x.reshape(shape + (comp, R)), Vs, per)).reshape(-1, R) - b * x) / a
    return apply


def _moments(op, r, M):
    """mu (R, M) of the start block r by the doubling identities."""
    dot = lambda u, v: (u.conj() * v).real.sum(dim=0)  # noqa: E731
    mu = torch.empty((r.shape[1], M + 1), dtype=torch.float64, device=r.device)
    prev, cur = r, op(r)
    mu[:, 0], mu[:, 1] = dot(r, r), dot(cur, r)
    for k in range(1, (M + 1) // 2):
        nxt = 2.0 * op(cur) - prev
        mu[:, 2 * k] = 2.0 * dot(cur, cur) - mu[:, 0]
        mu[:, 2 * k + 1] = 2.0 * dot(nxt, cur) - mu[:, 1]
        prev, cur = cur, nxt
    return mu[:, :M].contiguous()


def _series(op, x, c):
    out = c[0] * x
    if len(c) == 1:
        return out
    prev, cur = x, op(x)
    out = out + c[1] * cur
    for k in range(2, len(c)):
        prev, cur = cur, 2.0 * op(cur) - prev
        out = out + c[k] * cur
    return out


def _bessel(x: float, n: int) -> np.ndarray:
    """J_0..J_n(x): the periodic trapezoid rule on Bessel's integral, exact to rounding."""
    th = 2.0 * math.pi * np.arange(512) / 512
    return np.array([np.mean(np.cos(k * th - x * np.sin(th))) for k in range(n + 1)])


def _step_weights(case):
    """Chebyshev weights of exp(-i H dt), dt = 1, and its phase."""
    a, b = _scaling(case)
    J = _bessel(a, 40)
    last = max(k for k in range(41) if abs(J[k]) >= 1e-14)
    return [(1.0 if k == 0 else 2.0) * (-1j) ** k * float(J[k]) for k in range(last + 1)], np.exp(-1j * b)


def _mix(z: np.ndarray) -> np.ndarray:
    """SplitMix64's output function on uint64 arrays."""
    z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
    z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
    return z ^ (z >> np.uint64(31))


def _hashed_phases(D: int, R: int, seed: int) -> torch.Tensor:
    """The random-phase block that a call makes from a seed: exp(2 pi i u)/sqrt(D), u from the counter hash."""
    with np.errstate(over="ignore"):
        key = _mix(np.array([seed], dtype=np.uint64) ^ np.uint64(0x9E3779B97F4A7C15))
        h = _mix(key + np.arange(D * R, dtype=np.uint64))  # index r D + i
    u = torch.from_numpy(((h >> np.uint64(11)).astype(np.float64) * 2.0 ** -53).reshape(R, D).T.copy()).to(_dev())
    return torch.polar(torch.full_like(u, 1.0 / math.sqrt(D)), 2.0 * math.pi * u)


def _jackson(M: int) -> torch.Tensor:
    k = torch.arange(M, dtype=torch.float64, device=_dev())
    q = math.pi / (M + 1)
    return ((M - k + 1) * torch.cos(q * k) + torch.sin(q * k) / math.tan(q)) / (M + 1)


def exact(case, seed):
    kind = case["kind"]
    if kind == "batched":
        mus = []
        a, b = _batch_scaling(case)
        for i, (L, V) in enumerate(_cubes(case, seed)):
            one = {"kind": "kpm", "nx": L, "ny": L, "nz": L, "px": 1, "py": 1, "pz": 1, "W": case["W"]}
            r = _hashed_phases(4 * L ** 3, case["R"], int(seed) * 1000 + i)
            mus.append(_moments(_operator(one, V), r, case["M"]))
        return torch.stack(mus)
    if kind in ("propagate", "gradient"):
        V, psi = _dot_potential(case), _packets(case, seed)
        cw, phase = _step_weights(case)
        if kind == "propagate":
            x = psi.reshape(-1, case["R"])
            for _ in range(case["steps"]):
                x = complex(phase) * _series(_operator(case, V), x, cw)
            return x.reshape(psi.shape)
        V.requires_grad_(True)
        psi.requires_grad_(True)
        x = psi.reshape(-1, 1)
        for _ in range(case["steps"]):
            x = complex(phase) * _series(_operator(case, V), x, cw)
        x = x.reshape(-1)
        loss = (x.abs() ** 2 * _detector(case)).sum()
        gV, gpsi = torch.autograd.grad(loss, (V, psi))
        return {"loss": loss.detach(), "psi": x.detach(), "gV": gV, "gpsi": gpsi}
    V = _box(math.prod(_dims(case)), case["W"], seed) if case["W"] else None
    op = _operator(case, V)
    D = math.prod(_dims(case)) * _orbitals(case)
    if kind == "kpm":
        return _moments(op, _phases(D, case["R"], VEC[case["prec"]], seed).to(torch.complex128), case["M"])
    if kind == "step":
        x = _phases(D, case["R"], VEC[case["prec"]], seed).to(torch.complex128)
        y = op(x)
        xy = (y.conj() * x).sum(dim=0)
        return {"y": y, "dots": torch.stack([(x.abs() ** 2).sum(dim=0), xy.real, xy.imag, (y.abs() ** 2).sum(dim=0)])}
    if kind == "filter":
        return _series(op, _phases(D, case["R"], torch.complex128, seed), _filter_weights(case["K"]))
    # spectral: the four Bloch states of every k-point, Jackson-damped moments, summed per k-point
    nx, ny, nz = _dims(case)
    d = {"device": _dev(), "dtype": torch.float64}
    px = torch.arange(nx, **d)[None, None, :]
    py = torch.arange(ny, **d)[None, :, None]
    pz = torch.arange(nz, **d)[:, None, None]
    a, b = _scaling(case)
    E, g, out = _energies(case), _jackson(case["M"]), []
    th = torch.acos((E - b) / a)
    T = torch.cos(torch.arange(case["M"], **d)[:, None] * th[None, :])
    for k in _k_points(case, seed):
        arg = k[0] * px + k[1] * py + k[2] * pz
        wave = torch.polar(torch.full_like(arg, 1.0 / math.sqrt(nx * ny * nz)), arg).reshape(-1)
        psi = torch.zeros((wave.numel(), 4, 4), dtype=torch.complex128, device=wave.device)
        for o in range(4):
            psi[:, o, o] = wave
        mu = _moments(op, psi.reshape(-1, 4), case["M"]).sum(dim=0)
        w = g * mu
        out.append((w[0] + 2.0 * (w[1:, None] * T[1:]).sum(dim=0)) / (math.pi * a * torch.sin(th)))
    return torch.stack(out)
