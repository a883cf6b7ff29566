"""Performance cases of the lattice Boltzmann library, each through its public entry points.

A case advances one lattice (kind "single"), a batch of lattices ("batch"), or takes the
gradient of the objective ("adjoint"), or evaluates the observables of a state
("observe"), and returns everything the calls compute: fields, trace rows, energies,
gradients. Sizes and couplings are the ones of this repository's benchmark, experiments
and tests; draw() spreads over the same ranges. Inputs are the noisy uniform densities
every run of the model starts from (mean 0.7 or ln 2, +-1%), made on the GPU from the
seed. exact() evaluates the same definitions in 64 bits with plain torch operations.
"""
import math

import numpy as np
import torch
import torch.utils.checkpoint

from paper_1008_2865_gb300 import Batch, Lattice, couplings_from_A

BATCH_SIZES = (192, 384, 640)                          # the uneven sweep's lattice sizes
A2_SCAN = (-4.9, -2.85, -0.8, 0.15, 0.65, 1.15, 1.65, 2.15, 2.65)   # at A1 = -4.9

# Work of one site and step that no implementation can leave out (omega = 1): 46 FP
# operations for the force sums, 18 for the moments, 60 for the collision, 6 for the
# new density and about 20 for the exponential of psi.
STEP_FLOPS = 150
# One reverse step on top of a forward one: collision, force and stencil transposes.
REVERSE_FLOPS = 350


def _single(name, nx, ny, steps, prec="fp32", G1=-5.0, G2=0.6, omega=1.0, trace=10):
    return {"name": name, "kind": "single", "nx": nx, "ny": ny, "steps": steps, "prec": prec,
            "G1": G1, "G2": G2, "omega": omega, "trace": trace}


def listed():
    return [
        # smoke-sized lattice, ragged in both directions: the call is launches and latency
        _single("tiny 70x45", 70, 45, 100),
        # the FP64 parity run of the model (128^2, G2 = 0.5, trace every 10 steps)
        _single("fp64 128", 128, 128, 100, prec="fp64", G2=0.5),
        # a small study at another relaxation rate, no dimension a multiple of a tile
        _single("ragged 250x187 omega 0.8", 250, 187, 100, G2=0.3, omega=0.8),
        # the forward run behind the gradient workload: no trace
        _single("plain 512", 512, 512, 200, G2=0.5, trace=0),
        # one lattice of the 1024^2 coupling sweep: trace every 100 steps, fits in L2
        _single("sweep 1024", 1024, 1024, 100, trace=100),
        # a box just above L2 with ragged strips and rows
        _single("ragged 2050x1999", 2050, 1999, 40),
        # the benchmark's bandwidth run, FP32 storage
        _single("bench 8192", 8192, 8192, 20),
        # the same with FP16 storage of the deviations
        _single("fp16 8192", 8192, 8192, 20, prec="fp16_delta"),
        # the uneven 96-replica coupling sweep (32 each of 192^2, 384^2, 640^2)
        {"name": "batch 96 uneven", "kind": "batch", "set": "uneven", "count": 96, "n": 640,
         "steps": 100, "prec": "fp32", "trace": 10},
        # the A2 scan of the paper: nine 512^2 lattices from the plain model to the emulsions
        {"name": "batch A2 scan 9x512", "kind": "batch", "set": "scan", "count": 9, "n": 512,
         "steps": 200, "prec": "fp32", "trace": 1000},
        # the gradient workload: 512^2, 2000 steps, checkpoints every ceil(sqrt(T)) steps
        {"name": "adjoint 512 T 2000", "kind": "adjoint", "nx": 512, "ny": 512, "steps": 2000,
         "G1": -5.0, "G2": 0.5, "omega": 1.0},
        # what an analysis reads of a state: energies, objective and fields
        {"name": "observe 4096", "kind": "observe", "nx": 4096, "ny": 4096, "steps": 2,
         "prec": "fp32", "G1": -5.0, "G2": 0.6, "omega": 1.0},
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    """One more case: the kind by how often such calls are made, sizes log-uniform over the
    listed range with odd ones among them, steps so that no case is larger than the largest."""
    kind = rng.choices(["single", "batch", "adjoint", "observe"], [6, 2, 1, 1])[0]
    omega = rng.choice([1.0, 1.0, 1.0, round(rng.uniform(0.6, 1.4), 2)])
    G2 = round(rng.uniform(0.0, 0.9), 3)
    if kind == "single":
        prec = rng.choices(["fp32", "fp16_delta", "fp64"], [7, 2, 1])[0]
        hi = 512 if prec == "fp64" else 8192
        nx = _log_int(rng, 8, hi)
        ny = _log_int(rng, max(5, nx // 4), min(hi, 4 * nx))
        steps = max(10, min(200, int(8e8 / (nx * ny)))) if prec != "fp64" else 40
        steps = max(10, steps - rng.randrange(0, 10))
        return {"kind": kind, "nx": nx, "ny": ny, "steps": steps, "prec": prec, "G1": -5.0,
                "G2": G2, "omega": omega, "trace": rng.choice([0, 10, 10, 100])}
    if kind == "batch":
        which = rng.choice(["uneven", "scan"])
        n = _log_int(rng, 64, 640)
        count = rng.randrange(3, 97) if which == "uneven" else len(A2_SCAN)
        steps = max(10, min(200, int(1.5e9 / (count * n * n))))
        return {"kind": kind, "set": which, "count": count, "n": n, "steps": steps,
                "prec": rng.choice(["fp32", "fp32", "fp16_delta"]),
                "trace": rng.choice([10, 20, 1000])}
    nx = _log_int(rng, 32, 512 if kind == "adjoint" else 4096)
    ny = _log_int(rng, max(32, nx // 2), min(2 * nx, 512 if kind == "adjoint" else 4096))
    if kind == "adjoint":
        return {"kind": kind, "nx": nx, "ny": ny, "steps": _log_int(rng, 20, 400), "G1": -5.0,
                "G2": G2, "omega": omega}
    return {"kind": kind, "nx": nx, "ny": ny, "steps": 2,
            "prec": rng.choice(["fp32", "fp32", "fp16_delta"]), "G1": -5.0, "G2": G2,
            "omega": omega}


def _noise(nx, ny, seed, mean=0.7, amp=0.01):
    """Density mean (1 + amp U(-1, 1)) as [ny, nx] doubles on the GPU."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    u = torch.rand((ny, nx), generator=g, device="cuda", dtype=torch.float64)
    return u.mul_(2.0 * amp * mean).add_(mean * (1.0 - amp))


def _replicas(case, seed):
    """The batch's (nx, ny, G1, G2, initial density) per replica."""
    n, count = case["n"], case["count"]
    if case["set"] == "scan":
        pairs = [couplings_from_A(-4.9, a2) for a2 in A2_SCAN[:count]]
        return [(n, n, g1, g2, _noise(n, n, seed * 1000 + i, mean=math.log(2.0)))
                for i, (g1, g2) in enumerate(pairs)]
    sizes = [max(8, n * BATCH_SIZES[(3 * i) // count] // BATCH_SIZES[-1]) for i in range(count)]
    return [(m, m, -5.0, (i * 0.618034) % 1.0, _noise(m, m, seed * 1000 + i))
            for i, m in enumerate(sizes)]


def _stream():
    return torch.cuda.current_stream().cuda_stream


def _outputs(ny, nx):
    return [torch.empty((ny, nx), dtype=torch.float64, device="cuda") for _ in range(3)]


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        reps = _replicas(case, seed)
        b = Batch([r[4] for r in reps], G1=[r[2] for r in reps], G2=[r[3] for r in reps],
                  prec=case["prec"], trace_every=case["trace"], stream=_stream())
        flat = [torch.empty(sum(r[0] * r[1] for r in reps), dtype=torch.float64, device="cuda")
                for _ in range(3)]
        at = np.cumsum([0] + [r[0] * r[1] for r in reps])
        views = [[f[at[i]:at[i + 1]] for f in flat] for i in range(len(reps))]
        return {"case": case, "batch": b, "flat": flat, "views": views}
    nx, ny = case["nx"], case["ny"]
    rho = _noise(nx, ny, seed)
    if kind == "adjoint":
        return {"case": case, "rho": rho, "target": _noise(nx, ny, seed + 500000)}
    lat = Lattice(rho, omega=case["omega"], G1=case["G1"], G2=case["G2"], prec=case["prec"],
                  trace_every=case.get("trace", 0), stream=_stream())
    state = {"case": case, "lat": lat, "out": _outputs(ny, nx)}
    if kind == "observe":
        state["target"] = _noise(nx, ny, seed + 500000)
        lat.step(case["steps"])
    return state


def _trace_rows(case):
    return case["steps"] // case["trace"] if case["trace"] else 0


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "adjoint":
        # as the autograd wrapper does it: a fresh state, then the reverse sweep
        grad = torch.empty_like(state["rho"])
        with Lattice(state["rho"], omega=case["omega"], G1=case["G1"], G2=case["G2"],
                     trace_every=0, stream=_stream()) as lat:
            J, _, gG = lat.adjoint(case["steps"], state["target"], grad_rho=grad)
        return {"J": J, "grad": grad, "dG": list(gG)}
    if kind == "batch":
        b = state["batch"]
        b.step(case["steps"])
        for i, (rho, ux, uy) in enumerate(state["views"]):
            b.fields(i, rho, ux, uy)
        out = {"rho": state["flat"][0], "ux": state["flat"][1], "uy": state["flat"][2]}
        if _trace_rows(case):
            out["trace"] = np.concatenate([b.trace(i, _trace_rows(case)) for i in range(len(b))])
        return out
    lat = state["lat"]
    rho, ux, uy = state["out"]
    if kind == "observe":
        energy = lat.energy()
        J = lat.objective(state["target"])
        lat.fields(rho, ux, uy)
        return {"energy": list(energy), "J": J, "rho": rho, "ux": ux, "uy": uy}
    lat.step(case["steps"])
    lat.fields(rho, ux, uy)
    out = {"rho": rho, "ux": ux, "uy": uy}
    if _trace_rows(case):
        out["trace"] = lat.trace(_trace_rows(case))
    return out


def _state_bytes(case):
    return {"fp32": 40, "fp16_delta": 22, "fp64": 72}[case.get("prec", "fp32")]


def work(case):
    """Bytes: the state read and written once per pass and the outputs written once (a pass of
    many steps need not go back to memory between them); FP operations of every step."""
    kind = case["kind"]
    if kind == "batch":
        n, count = case["n"], case["count"]
        if case["set"] == "scan":
            sites = count * n * n
        else:
            sites = sum(max(8, n * BATCH_SIZES[(3 * i) // count] // BATCH_SIZES[-1]) ** 2
                        for i in range(count))
    else:
        sites = case["nx"] * case["ny"]
    if kind == "adjoint":
        # rho_init and the target read, the gradient written
        return {"bytes": 24 * sites,
                "flops": sites * case["steps"] * (STEP_FLOPS + REVERSE_FLOPS)}
    if kind == "observe":
        # the state for the energies and the fields, the target, three fields written
        return {"bytes": sites * (_state_bytes(case) + 8 + 24), "flops": 120 * sites}
    return {"bytes": sites * (2 * _state_bytes(case) + 24),
            "flops": sites * case["steps"] * STEP_FLOPS}


# ---- the same definitions in 64 bits, with torch operations only

_C = [(0, 0), (1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, 1), (-1, -1), (1, -1)]
_W = [4 / 9] + [1 / 9] * 4 + [1 / 36] * 4
_P = {1: 4 / 63, 2: 4 / 135, 4: 1 / 180, 5: 2 / 945, 8: 1 / 15120}   # mid-range weights by |c|^2
_LINKS = [(cx, cy) for cx in range(-2, 3) for cy in range(-2, 3) if (cx, cy) != (0, 0)]


def _at(v, cx, cy):
    """v(x + c) on the periodic lattice [..., y, x]."""
    return torch.roll(v, (-cy, -cx), (-2, -1))


def _link(cx, cy, G1, G2):
    c2 = cx * cx + cy * cy
    return (G1 * _W[1 if c2 == 1 else 5] if c2 <= 2 else 0.0) + G2 * _P[c2]


def _psi(rho):
    return -torch.expm1(-rho)


def _moments(f):
    rho = sum(f)
    ux = sum(c[0] * fi for c, fi in zip(_C, f) if c[0]) / rho
    uy = sum(c[1] * fi for c, fi in zip(_C, f) if c[1]) / rho
    return rho, ux, uy


def _step(f, G1, G2, omega):
    rho, ux, uy = _moments(f)
    psi = _psi(rho)
    sx, sy = torch.zeros_like(rho), torch.zeros_like(rho)
    for cx, cy in _LINKS:
        p = _link(cx, cy, G1, G2) * _at(psi, cx, cy)
        if cx:
            sx = sx + cx * p
        if cy:
            sy = sy + cy * p
    vx, vy = ux - psi * sx / (omega * rho), uy - psi * sy / (omega * rho)
    sq = 1.5 * (vx * vx + vy * vy)
    out = []
    for (cx, cy), w, fi in zip(_C, _W, f):
        cu = cx * vx + cy * vy
        feq = w * rho * (1 + 3 * cu + 4.5 * cu * cu - sq)
        out.append(_at((1 - omega) * fi + omega * feq, -cx, -cy))
    return out


def _energies(rho, G1, G2):
    """(mass, E_s, E_m, E_bulk) over the last two dimensions."""
    psi = _psi(rho)
    p0 = 1 - 4 * (_P[1] + _P[2] + _P[4] + 2 * _P[5] + _P[8])
    s, m = (G1 * _W[0] + G2 * p0) * psi, torch.zeros_like(psi)
    for cx, cy in _LINKS:
        p = _link(cx, cy, G1, G2) * _at(psi, cx, cy)
        if cx * cx + cy * cy <= 2:
            s = s + p
        else:
            m = m + p
    return [v.sum((-2, -1)) for v in (rho, 0.5 * psi * s, 0.5 * psi * m,
                                      0.5 * (G1 + G2) * psi * psi)]


def _run64(rho, G1, G2, omega, steps, trace):
    f = [w * rho for w in _W]
    rows = []
    for t in range(steps):
        if trace and t % trace == 0:
            rows.append((t, _energies(sum(f), G1, G2)))
        f = _step(f, G1, G2, omega)
    return f, rows


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        reps = _replicas(case, seed)
        found = [None] * len(reps)
        for size in sorted({r[:2] for r in reps}):          # replicas of one size side by side
            ids = [i for i, r in enumerate(reps) if r[:2] == size]
            G1, G2 = (torch.tensor([reps[i][k] for i in ids], dtype=torch.float64,
                                   device="cuda").view(-1, 1, 1) for k in (2, 3))
            f, rows = _run64(torch.stack([reps[i][4] for i in ids]), G1, G2, 1.0, case["steps"],
                             case["trace"])
            mom = _moments(f)
            for j, i in enumerate(ids):
                tr = np.array([[t] + [float(e[j]) for e in es] for t, es in rows])
                found[i] = ([m[j].reshape(-1) for m in mom], tr)
        out = {k: torch.cat([r[0][q] for r in found]) for q, k in enumerate(("rho", "ux", "uy"))}
        if _trace_rows(case):
            out["trace"] = np.concatenate([r[1][-_trace_rows(case):] for r in found])
        return out
    nx, ny, G1, G2, omega, steps = (case[k] for k in ("nx", "ny", "G1", "G2", "omega", "steps"))
    rho = _noise(nx, ny, seed)
    if kind == "adjoint":
        if nx * ny * steps > 512 * 512 * 100:
            return None                                     # minutes and too much memory
        target = _noise(nx, ny, seed + 500000)
        rho.requires_grad_(True)
        g = [torch.tensor(v, dtype=torch.float64, device="cuda", requires_grad=True)
             for v in (G1, G2)]
        f = [w * rho for w in _W]
        for _ in range(steps):
            f = list(torch.utils.checkpoint.checkpoint(
                lambda *v: tuple(_step(list(v), g[0], g[1], omega)), *f, use_reentrant=False))
        r = sum(f)
        _, es, em, _ = _energies(r, g[0], g[1])
        J = es + em + (r - target).square().sum()
        gr, g1, g2 = torch.autograd.grad(J, [rho] + g)
        return {"J": float(J), "grad": gr, "dG": [float(g1), float(g2)]}
    f, rows = _run64(rho, G1, G2, omega, steps, case.get("trace", 0))
    r, ux, uy = _moments(f)
    if kind == "observe":
        mass, es, em, eb = (float(v) for v in _energies(r, G1, G2))
        J = es + em + float((r - _noise(nx, ny, seed + 500000)).square().sum())
        return {"energy": [es, em, eb, mass], "J": J, "rho": r, "ux": ux, "uy": uy}
    out = {"rho": r, "ux": ux, "uy": uy}
    if _trace_rows(case):
        tr = np.array([[t] + [float(e) for e in es] for t, es in rows])
        out["trace"] = tr[-_trace_rows(case):]
    return out
