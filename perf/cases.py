"""Performance cases: what a user of the hard-disk library has it do.

Chains (kinds "probe", "run", "scan"): a context started on its lattice and
relaxed for some sweeps, then one pass of the work a simulation repeats --
bursts of sweeps with an acceptance read-back, steps of sweeps with the
pressure and Psi_6 measured on the device and read back, a whole
equation-of-state scan in one context.  Snapshots (kinds "snapshot",
"pressure", "corr", "sq"): a configuration the user holds, analysed through
the measurement calls.  "tau": the correlation time of a recorded series.

`exact` restates the snapshot analyses in 64 bits from the configuration's
own lattice indices; a chain, and the configuration of "pressure" that a
chain relaxed, have no such value.
"""
import math

import numpy as np
import torch

import paper_1211_1645_gb300 as hd

FX = 16777216.0  # fixed-point units per sigma


def listed():
    return [
        # Acceptance probing of a small ragged system (what tuning the step
        # size repeats): 20 sweeps, then the trial counts.
        {"name": "probe_n1000_fixed", "kind": "probe", "N": 1000, "eta": 0.70, "precision": "fixed", "sweeps": 20},
        # The 256-disk system of configuration 1 (N = 16^2, eta = 0.70, plain
        # FP64): ten steps of 100 sweeps, each measured.
        {"name": "run_n256_fp64", "kind": "run", "N": 256, "eta": 0.70, "precision": "fp64", "steps": 10,
         "sweeps": 100, "measure": 1, "lattice": "square"},
        # Configuration 2 (N = 256^2, eta = 0.708): a step of 100 sweeps and a measurement.
        {"name": "run_n65536_fixed", "kind": "run", "N": 65536, "eta": 0.708, "precision": "fixed", "steps": 1,
         "sweeps": 100, "measure": 1, "lattice": "square"},
        # The benchmark's system (N = 1024^2, eta = 0.716), both number forms.
        {"name": "run_n1m_fixed", "kind": "run", "N": 1048576, "eta": 0.716, "precision": "fixed", "steps": 1,
         "sweeps": 100, "measure": 1, "lattice": "square"},
        {"name": "run_n1m_fp64", "kind": "run", "N": 1048576, "eta": 0.716, "precision": "fp64", "steps": 1,
         "sweeps": 100, "measure": 1, "lattice": "square"},
        # Configuration 5 (N = 2048^2, eta = 0.720, shifted rows): 250 sweeps
        # and a measurement that keeps the local psi_j field.
        {"name": "run_n4m_field_fixed", "kind": "run", "N": 4194304, "eta": 0.720, "precision": "fixed", "steps": 1,
         "sweeps": 250, "measure": 2, "lattice": "triangular"},
        # The 31-replica equation-of-state scan (N = 128^2 .. 512^2, eta = 0.700 + 0.001 r).
        {"name": "scan31_fixed", "kind": "scan", "R": 31, "base": 128, "precision": "fixed", "sweeps": 100},
        # A stored configuration brought in and its local and coarse psi_6
        # fields (sampling areas of ten disks) taken out.
        {"name": "snapshot_n262144_fixed", "kind": "snapshot", "N": 262144, "eta": 0.716, "precision": "fixed",
         "bins": 162},
        # A stored configuration's contact pressure, and its positions read back, plain FP64.
        {"name": "pressure_n1m_fp64", "kind": "pressure", "N": 1048576, "eta": 0.716, "precision": "fp64"},
        # Positional order of a solid-like configuration: q_0, the chi field
        # and the correlation function out to 20 sigma.
        {"name": "corr_n16384_fixed", "kind": "corr", "N": 16384, "eta": 0.720, "precision": "fixed", "nr": 40,
         "dr": 0.5, "half_width": 3, "bins": 32},
        # The structure factor over a map of wave vectors around the first shell.
        {"name": "sq_n65536_fp64", "kind": "sq", "N": 65536, "eta": 0.716, "precision": "fp64", "side": 21},
        # Psi_6 autocorrelation and correlation time of four recorded chains.
        {"name": "tau_t4000_fixed", "kind": "tau", "N": 64, "eta": 0.65, "precision": "fixed", "R": 4, "T": 4000,
         "max_lag": 400},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["probe", "run", "run", "run", "run", "scan", "snapshot", "pressure", "corr", "sq", "tau"])
    precision = rng.choice(["fixed", "fp64"])
    eta = round(rng.uniform(0.65, 0.73), 3)
    if kind == "probe":
        N = _log_int(rng, 200, 100000)
        # a small ragged count needs a thinner system for its square start lattice to fit
        return {"kind": kind, "N": N, "eta": eta if N >= 1000 else 0.65, "precision": precision,
                "sweeps": rng.choice([5, 10, 20, 40])}
    if kind == "run":
        N = _log_int(rng, 200, 2000000)
        return {"kind": kind, "N": N, "eta": eta if N >= 1000 else 0.65, "precision": precision,
                "steps": rng.choice([1, 2, 5]) if N < 100000 else 1,
                "sweeps": rng.choice([25, 50, 100, 101]), "measure": rng.choice([0, 1, 1, 2]),
                "lattice": rng.choice(["square", "triangular"])}
    if kind == "scan":
        return {"kind": kind, "R": rng.randint(2, 31), "base": _log_int(rng, 16, 128), "precision": precision,
                "sweeps": rng.choice([20, 50, 100])}
    if kind == "snapshot":
        N = _log_int(rng, 1000, 600000)
        return {"kind": kind, "N": N, "eta": eta, "precision": precision, "bins": max(4, int(math.sqrt(N / rng.uniform(5, 20))))}
    if kind == "pressure":
        return {"kind": kind, "N": _log_int(rng, 1000, 1500000), "eta": eta, "precision": precision}
    if kind == "corr":
        N = _log_int(rng, 2500, 16384)
        return {"kind": kind, "N": N, "eta": eta, "precision": precision, "nr": rng.choice([20, 33, 40]),
                "dr": rng.choice([0.25, 0.4, 0.5]), "half_width": rng.choice([2, 3, 4]),
                "bins": max(4, int(math.sqrt(N / rng.uniform(5, 20))))}
    if kind == "sq":
        return {"kind": kind, "N": _log_int(rng, 1000, 100000), "eta": eta, "precision": precision,
                "side": rng.choice([5, 9, 14, 21])}
    return {"kind": kind, "N": rng.choice([64, 81, 100]), "eta": round(rng.uniform(0.5, 0.66), 3),
            "precision": precision, "R": rng.randint(1, 6), "T": _log_int(rng, 300, 4000), "max_lag": rng.randint(20, 250)}


# ---------------------------------------------------------------------------
# Configurations: a triangular lattice fitted to the square box (even number
# of rows, odd rows shifted), surplus sites vacant, each disk displaced at
# random by less than half the gap, ids in random order.
# ---------------------------------------------------------------------------
def _lattice_shape(case):
    N = case["N"]
    L = math.sqrt(N * math.pi / case["eta"])
    ny = 2 * int(round(math.sqrt(2.0 * N / math.sqrt(3.0)) / 2.0))
    nx = -(-N // ny)
    return L, nx, ny


def _sites(case, seed):
    """x, y (FP64) and the disk id (-1: vacant) of every lattice site [ny, nx]."""
    N = case["N"]
    L, nx, ny = _lattice_shape(case)
    dx, dy = L / nx, L / ny
    gap = min(dx, math.hypot(0.5 * dx, dy)) - 2.0
    g = torch.Generator(device="cuda")
    g.manual_seed(1000003 * int(seed) + N)
    kw = {"generator": g, "device": "cuda"}
    row = torch.arange(ny, device="cuda", dtype=torch.float64)[:, None]
    col = torch.arange(nx, device="cuda", dtype=torch.float64)[None, :]
    amp = 0.49 * max(gap, 0.0) * torch.sqrt(torch.rand((ny, nx), dtype=torch.float64, **kw))
    ang = 2.0 * math.pi * torch.rand((ny, nx), dtype=torch.float64, **kw)
    x = (col + 0.5 * torch.remainder(row, 2.0) + 0.25) * dx + amp * torch.cos(ang)
    y = (row + 0.5) * dy + amp * torch.sin(ang)
    ids = torch.full((ny * nx,), -1, dtype=torch.int64, device="cuda")
    order = torch.randperm(ny * nx, **kw)
    ids[order[:N]] = torch.arange(N, device="cuda")
    return torch.remainder(x, L), torch.remainder(y, L), ids.view(ny, nx), L


def _positions(case, seed):
    """The configuration as the user holds it: pinned host memory, [N, 2] by disk id."""
    x, y, ids, _ = _sites(case, seed)
    keep = ids >= 0
    xy = torch.empty((case["N"], 2), dtype=torch.float64, device="cuda")
    xy[ids[keep], 0] = x[keep]
    xy[ids[keep], 1] = y[keep]
    out = torch.empty((case["N"], 2), dtype=torch.float64, pin_memory=True)
    out.copy_(xy)
    return out


def _wave_vectors(case):
    """side x side box wave vectors around a first-shell reciprocal vector of the lattice."""
    L, nx, ny = _lattice_shape(case)
    s = case["side"]
    h, k = np.meshgrid(np.arange(s) - s // 2 + nx, np.arange(s) - s // 2 + ny // 2, indexing="ij")
    return np.stack([h.ravel(), k.ravel()], axis=1).astype(np.int32)


SCAN_N = [1.0, 1.5, 2.0, 3.0, 4.0]  # replica sides in units of the scan's smallest


def _scan(case):
    R = case["R"]
    Ns = [int(case["base"] * SCAN_N[r % 5]) ** 2 for r in range(R)]
    return Ns, [0.700 + 0.001 * r for r in range(R)]


def prepare(case, seed):
    kind, form = case["kind"], case["precision"]
    if kind == "scan":
        Ns, etas = _scan(case)
        g = hd.HardDisks(Ns, etas, [0.1] * len(Ns), [seed * 1000 + r + 1 for r in range(len(Ns))], precision=form)
        g.sweep(50)
        return {"case": case, "g": g, "xy": torch.empty((sum(Ns), 2), dtype=torch.float64, device="cuda")}
    if kind == "tau":
        R = case["R"]
        g = hd.HardDisks([case["N"]] * R, [case["eta"]] * R, [0.2] * R, [seed * 1000 + r + 1 for r in range(R)],
                         precision=form)
        g.series_reserve(case["T"])
        g.run(case["T"], 1, True)
        return {"case": case, "g": g}
    g = hd.HardDisks(case["N"], case["eta"], 0.1, seed + 1, precision=form, lattice=case.get("lattice", "square"))
    if kind in ("probe", "run"):
        g.sweep(50 if case["N"] > 10 ** 5 else 400)
        return {"case": case, "g": g, "xy": torch.empty((case["N"], 2), dtype=torch.float64, device="cuda"),
                "psi": torch.empty((case["N"], 2), dtype=torch.float64, device="cuda")}
    host = _positions(case, seed)
    state = {"case": case, "g": g, "host": host, "np": host.numpy()}
    if kind != "snapshot":
        g.set_positions(state["np"])
    if kind == "pressure":  # a liquid's contact shell: let the chain fill it, and store that configuration
        g.sweep(50)
        state["np"][:] = g.positions()
    if kind == "sq":
        state["hk"] = _wave_vectors(case)
    return state


def run(state):
    case, g = state["case"], state["g"]
    kind = case["kind"]
    if kind == "probe":
        g.sweep(case["sweeps"])
        att, acc = g.stats()
        hd.hd_positions_device(g.h, state["xy"].data_ptr())
        return {"attempts": att.astype(np.int64), "accepts": acc.astype(np.int64), "xy": state["xy"]}
    if kind in ("run", "scan"):
        g.run(case.get("steps", 1), case["sweeps"], case.get("measure", 1))
        out = {"xy": state["xy"]}
        hd.hd_positions_device(g.h, state["xy"].data_ptr())
        if case.get("measure", 1):
            out["series"] = g.series()
            g.series_clear()
        if case.get("measure", 1) == 2:
            g.psi6_local_device(state["psi"].data_ptr())
            out["psi"] = state["psi"]
        return out
    if kind == "snapshot":
        g.set_positions(state["np"])
        psi, local = g.psi6()
        return {"psi": psi, "local": local, "field": g.psi6_field(case["bins"])}
    if kind == "pressure":
        g.set_positions(state["np"])
        bp, g0, hist = g.pressure()
        return {"bp": bp, "g0": g0, "hist": hist.astype(np.int64), "xy": g.positions()}
    if kind == "corr":
        hk0, S0 = g.positional_q0(case["half_width"])
        return {"hk0": hk0, "S0": S0, "chi": g.positional_field(hk0, case["bins"]),
                "C": g.positional_corr(hk0, case["nr"], case["dr"])}
    if kind == "sq":
        return {"S": g.structure_factor(state["hk"])}
    return {"acf": g.psi6_acf(case["max_lag"]), "tau": g.psi6_tau(1, 15), "series": g.series()}


def _state_bytes(N, form):
    return N * ((8 if form == "fixed" else 16) + 4)


def work(case):
    """Bytes: inputs and outputs once.  Operations: a trial move is ~100
    (generator block, step, ~8 pair distances), a pair or candidate ~10, a
    wave-vector phase ~40 per disk."""
    kind, form = case["kind"], case["precision"]
    if kind == "scan":
        N = sum(_scan(case)[0])
        return {"bytes": 2 * _state_bytes(N, form) + 16 * N, "flops": N * (100 * case["sweeps"] + 500)}
    N = case["N"]
    if kind == "probe":
        return {"bytes": 2 * _state_bytes(N, form) + 16 * N, "flops": 100 * N * case["sweeps"]}
    if kind == "run":
        b = 2 * _state_bytes(N, form) + 16 * N + (32 * N if case["measure"] == 2 else 0)
        return {"bytes": b, "flops": case["steps"] * N * (100 * case["sweeps"] + (500 if case["measure"] else 0))}
    if kind == "snapshot":
        return {"bytes": 16 * N + 16 * N + 16 * case["bins"] ** 2, "flops": 500 * N}
    if kind == "pressure":
        return {"bytes": 16 * N + 16 * N, "flops": 150 * N}
    if kind == "corr":
        pairs = N * case["eta"] * (case["nr"] * case["dr"] + 1.0) ** 2
        return {"bytes": _state_bytes(N, form), "flops": 10 * pairs + 40 * N * (2 * case["half_width"] + 1) ** 2}
    if kind == "sq":
        return {"bytes": _state_bytes(N, form), "flops": 40 * N * case["side"] ** 2}
    return {"bytes": 32 * case["R"] * case["T"], "flops": 8 * case["R"] * case["T"] * (case["max_lag"] + 16)}


# ---------------------------------------------------------------------------
# The snapshot analyses in 64 bits
# ---------------------------------------------------------------------------
def _box(case, L):
    """Cells per side, box side and (fixed form) cell side in units of 2^-24 sigma."""
    m = 2 * int(math.floor(L / 4.0))
    if case["precision"] == "fixed":
        W = int(round(L / m * FX))
        return m * W / FX, m * W
    return L, None


def _shifted(v, dr, dc):
    return torch.roll(v, shifts=(-dr, -dc), dims=(0, 1))


def _offsets(nx, ny, dx, dy, reach):
    """(row, column) site offsets whose disks can lie within `reach` of each other."""
    rr, cc = int(reach / dy) + 2, int(reach / dx) + 2
    rr, cc = min(rr, (ny - 1) // 2), min(cc, (nx - 1) // 2)
    return [(a, b) for a in range(-rr, rr + 1) for b in range(-cc, cc + 1) if (a, b) != (0, 0)]


def exact(case, seed):
    kind = case["kind"]
    if kind not in ("snapshot", "corr", "sq"):
        return None
    x, y, ids, L = _sites(case, seed)
    ny, nx = ids.shape
    dx, dy = L / nx, L / ny
    box, LF = _box(case, L)
    if LF is not None:  # the fixed form rounds to its grid and wraps into its own box
        x = torch.remainder(torch.round(x * FX), float(LF)) / FX
        y = torch.remainder(torch.round(y * FX), float(LF)) / FX
    here = ids >= 0

    def pair(a, b):
        ux, uy = _shifted(x, a, b) - x, _shifted(y, a, b) - y
        return ux - box * torch.round(ux / box), uy - box * torch.round(uy / box), here & _shifted(here, a, b)

    def by_id(v):
        out = torch.empty(case["N"], dtype=v.dtype, device=v.device)
        out[ids[here]] = v[here]
        return out

    def psi6():
        d2, vx, vy = [], [], []
        for a, b in _offsets(nx, ny, dx, dy, 2.0 * dx):
            ux, uy, both = pair(a, b)
            d2.append(torch.where(both, ux * ux + uy * uy, torch.inf))
            vx.append(ux)
            vy.append(uy)
        near = torch.topk(torch.stack(d2), 6, dim=0, largest=False).indices
        phi = torch.atan2(torch.stack(vy).gather(0, near), torch.stack(vx).gather(0, near))
        return torch.complex(torch.cos(6.0 * phi).mean(0), torch.sin(6.0 * phi).mean(0))

    def coarse(v, bins):
        ix = torch.clamp(torch.floor(x / box * bins).long(), max=bins - 1)
        iy = torch.clamp(torch.floor(y / box * bins).long(), max=bins - 1)
        at = (iy * bins + ix)[here]
        n = torch.zeros(bins * bins, dtype=torch.float64, device="cuda").index_add_(0, at, torch.ones_like(at, dtype=torch.float64))
        re = torch.zeros_like(n).index_add_(0, at, v.real[here])
        im = torch.zeros_like(n).index_add_(0, at, v.imag[here])
        return torch.complex(re / n, im / n).view(1, bins, bins).cpu().numpy()

    def amplitude(h, k):
        t = torch.remainder(h * (x[here] / box), 1.0) + torch.remainder(k * (y[here] / box), 1.0)
        return torch.complex(torch.cos(2.0 * math.pi * t), torch.sin(2.0 * math.pi * t)).sum()

    def S(hk):
        return np.array([[float((amplitude(int(h), int(k)).abs() ** 2).item()) / case["N"] for h, k in hk]])

    if kind == "snapshot":
        v = psi6()
        return {"psi": v[here].mean().view(1).cpu().numpy(), "local": by_id(v).cpu().numpy(),
                "field": coarse(v, case["bins"])}
    if kind == "sq":
        return {"S": S(_wave_vectors(case))}
    mean = psi6()[here].mean()
    a0 = math.sqrt(2.0 * box * box / (math.sqrt(3.0) * case["N"]))
    th = math.atan2(mean.imag.item(), mean.real.item()) / 6.0 + math.pi / 6.0
    q = 4.0 * math.pi / (a0 * math.sqrt(3.0)) * box / (2.0 * math.pi)
    w = case["half_width"]
    hk = [(int(round(q * math.cos(th))) + i, int(round(q * math.sin(th))) + j)
          for i in range(-w, w + 1) for j in range(-w, w + 1)]
    values = S(hk)[0]
    h, k = hk[int(np.argmax(values))]
    t = 2.0 * math.pi * (torch.remainder(h * (x / box), 1.0) + torch.remainder(k * (y / box), 1.0))
    chi = torch.complex(torch.cos(t), torch.sin(t))
    r = (torch.arange(case["nr"], dtype=torch.float64, device="cuda") + 1.0) * case["dr"]
    lo, hi = torch.clamp(r - 1.0, min=0.0)[:, None], (r + 1.0)[:, None]
    total = torch.zeros(case["nr"], dtype=torch.complex128, device="cuda")
    count = torch.zeros(case["nr"], dtype=torch.float64, device="cuda")
    for a, b in _offsets(nx, ny, dx, dy, case["nr"] * case["dr"] + 1.0):
        ux, uy, both = pair(a, b)
        d = torch.sqrt(ux * ux + uy * uy)[both][None, :]
        v = (chi * _shifted(chi, a, b).conj())[both][None, :]
        inside = (d >= lo) & (d <= hi)
        total += torch.where(inside, v, torch.zeros_like(v)).sum(1)
        count += inside.sum(1)
    C = torch.where(count > 0, total / count, torch.full_like(total, complex(math.nan, math.nan)))
    return {"hk0": None, "S0": np.array([float(values.max())]), "chi": coarse(chi, case["bins"]),
            "C": C.view(1, -1).cpu().numpy()}
