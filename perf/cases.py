"""Performance cases: what programs that use this library ask of it, through its public Python entry points.

A case is one kind of call on one state:

  sweep    Monte Carlo sweeps of one system or of a batch of replicas, then the energy and the state (the production run
           between two read-outs)
  restart  the same from host arrays: set_state, sweeps, energy, state (a driver program that owns the configuration)
  corr     sweeps with the many-origin time correlations on the way, then the statistics (the relaxation-time study)
  obs      F_s, F_s^cm and C_2 of every particle against one time origin
  static   the static analysis of a snapshot: S(q), g(r), virial pressure and energy
  md       molecular dynamics steps, then velocities, thermostat and positions

Systems are the paper's liquid at rho = 1.2, made from the seed: molecules with random orientations on a cubic lattice,
then Monte Carlo sweeps at the case's temperature.
"""
import math

import numpy as np
import torch

from paper_2506_21290_gb300 import flipmc as F
from paper_2506_21290_gb300 import speedup as SP
from paper_2506_21290_gb300 import workloads as W

MIXES = {"paper": W.PAPER_MIX, "local": W.LOCAL_MIX, "rigid": W.RIGID_MIX}
STATS = ("rejected_geometry", "rejected_bond", "pair_evals", "fp64_rechecks", "pair_interactions", "sweeps")


def listed():
    return [
        # the smallest system of the parity runs, FP64 chain, a handful of sweeps: launches and waits are all of it
        {"name": "sweep-64-fp64", "kind": "sweep", "R": 1, "M": 64, "M_hi": 64, "T": 3.0, "precision": "fp64",
         "mix": "paper", "sweeps": 5, "tune": 0, "recompute": 0},
        # one small system at an intermediate temperature, the production precision
        {"name": "sweep-1000", "kind": "sweep", "R": 1, "M": 1000, "M_hi": 1000, "T": 1.1, "precision": "fp32",
         "mix": "paper", "sweeps": 100, "tune": 0, "recompute": 0},
        # the headline system, at the lowest temperature, schedule picked by the autotuner as the benchmark does
        {"name": "sweep-8000", "kind": "sweep", "R": 1, "M": 8000, "M_hi": 8000, "T": 0.75, "precision": "fp32",
         "mix": "paper", "sweeps": 100, "tune": 20, "recompute": 0},
        # the headline system as the exact FP64 chain (reference trajectories, audits)
        {"name": "sweep-8000-fp64", "kind": "sweep", "R": 1, "M": 8000, "M_hi": 8000, "T": 0.75, "precision": "fp64",
         "mix": "paper", "sweeps": 20, "tune": 0, "recompute": 0},
        # the largest single system, with its drift check every 100 sweeps
        {"name": "sweep-64000", "kind": "sweep", "R": 1, "M": 64000, "M_hi": 64000, "T": 0.75, "precision": "fp32",
         "mix": "paper", "sweeps": 100, "tune": 0, "recompute": 100},
        # independent samples of uneven size and temperature advanced together
        {"name": "batch-256", "kind": "sweep", "R": 256, "M": 256, "M_hi": 2000, "T": 0.75, "precision": "fp32",
         "mix": "paper", "sweeps": 20, "tune": 8, "recompute": 0},
        # host arrays in, host arrays out, each step
        {"name": "restart-8000", "kind": "restart", "R": 1, "M": 8000, "M_hi": 8000, "T": 0.75, "precision": "fp32",
         "mix": "paper", "sweeps": 20, "tune": 0, "recompute": 0},
        # the relaxation-time study of flip against local moves: 8 replicas, log-spaced lags, 16 origins
        {"name": "corr-8x1000", "kind": "corr", "R": 8, "M": 1000, "T": 2.0, "mix": "paper", "lag_max": 2000,
         "origins": 16, "sweeps": 1000, "n_q": 48},
        # per-particle relaxation of one snapshot pair (mobility maps)
        {"name": "obs-8000", "kind": "obs", "R": 1, "M": 8000, "T": 1.1, "sweeps": 200, "n_q": 48},
        # static analysis of one snapshot: S(q) through its first peak, g(r) to half the box
        {"name": "static-8000", "kind": "static", "R": 1, "M": 8000, "T": 1.1, "n_q": 240, "bins": 280},
        # the paper's NVT molecular dynamics (time step 0.001, thermostat time 1), FP64 forces
        {"name": "md-1000-fp64", "kind": "md", "M": 1000, "T": 1.5, "tau": 1.0, "forces": "fp64", "steps": 50},
        # the same of the largest system with FP32 pair forces
        {"name": "md-64000-fp32", "kind": "md", "M": 64000, "T": 1.5, "tau": 1.0, "forces": "fp32", "steps": 50},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["sweep", "sweep", "sweep", "batch", "restart", "corr", "obs", "static", "md", "md"])
    T = round(rng.uniform(W.T_LOW, W.T_HIGH), 3)
    mix = rng.choice(["paper", "paper", "paper", "local", "rigid"])
    precision = rng.choice(["fp32", "fp32", "fp64"])
    if kind == "sweep":
        M = _log_int(rng, 64, 64000)
        return {"kind": "sweep", "R": 1, "M": M, "M_hi": M, "T": T, "precision": precision, "mix": mix,
                "sweeps": rng.randint(5, 20 if precision == "fp64" else 60), "tune": rng.choice([0, 0, 4]),
                "recompute": rng.choice([0, 0, 10])}
    if kind == "batch":
        lo = _log_int(rng, 64, 1200)
        return {"kind": "sweep", "R": _log_int(rng, 2, 150), "M": lo, "M_hi": rng.randint(lo, min(2 * lo, 2000)), "T": T,
                "precision": precision, "mix": mix, "sweeps": rng.randint(2, 4 if precision == "fp64" else 12),
                "tune": rng.choice([0, 0, 2]), "recompute": 0}
    if kind == "restart":
        M = _log_int(rng, 64, 20000)
        return {"kind": "restart", "R": 1, "M": M, "M_hi": M, "T": T, "precision": precision, "mix": mix,
                "sweeps": rng.randint(1, 20), "tune": 0, "recompute": 0}
    if kind == "corr":
        return {"kind": "corr", "R": _log_int(rng, 1, 8), "M": _log_int(rng, 64, 1200), "T": round(rng.uniform(1.4, 3.0), 3),
                "mix": rng.choice(["paper", "local"]), "lag_max": _log_int(rng, 16, 600), "origins": rng.randint(1, 16),
                "sweeps": rng.randint(20, 300), "n_q": rng.randint(6, 48)}
    if kind == "obs":
        return {"kind": "obs", "R": rng.randint(1, 4), "M": _log_int(rng, 64, 10000), "T": T, "sweeps": rng.randint(1, 300),
                "n_q": rng.randint(1, 64)}
    if kind == "static":
        return {"kind": "static", "R": rng.randint(1, 3), "M": _log_int(rng, 64, 6000), "T": T, "n_q": rng.randint(3, 240),
                "bins": _log_int(rng, 20, 800)}
    forces = rng.choice(["fp64", "fp32"])
    return {"kind": "md", "M": _log_int(rng, 64, 8000 if forces == "fp64" else 64000), "T": round(rng.uniform(1.2, 3.0), 3),
            "tau": rng.choice([1.0, 1.0, 0.0]), "forces": forces, "steps": rng.randint(5, 40)}


# --- the systems -----------------------------------------------------------------------------------------------------


def _molecule():
    """The A-B-C triangle with sides 0.96 sigma_ab, centroid at the origin."""
    a, b, c = W.SIGMA
    ab, bc, ac = (0.96 * 0.5 * (x + y) for x, y in ((a, b), (b, c), (a, c)))
    x = (ab * ab + ac * ac - bc * bc) / (2.0 * ab)
    tri = np.array([[0.0, 0.0, 0.0], [ab, 0.0, 0.0], [x, math.sqrt(ac * ac - x * x), 0.0]])
    return tri - tri.mean(axis=0)


def _start(M, L, rng):
    """M molecules of random orientation on the first points of a cubic lattice of the box."""
    m = max(1, math.ceil(M ** (1.0 / 3.0) - 1e-9))
    i = np.arange(M)
    centre = (np.stack([i % m, (i // m) % m, i // (m * m)], axis=1) + 0.5) * (L / m)
    a = rng.normal(size=(M, 3))
    a /= np.linalg.norm(a, axis=1, keepdims=True)
    b = rng.normal(size=(M, 3))
    b -= (a * b).sum(axis=1, keepdims=True) * a
    b /= np.linalg.norm(b, axis=1, keepdims=True)
    tri = _molecule()
    return (centre[:, None] + tri[None, :, :1] * a[:, None] + tri[None, :, 1:2] * b[:, None]).reshape(-1, 3)


def _system(sizes, T, seed, precision="fp32", recompute=0, n_eq=400):
    """A handle of replicas of the given sizes after n_eq sweeps at T (one value, or one per replica)."""
    rng = np.random.default_rng([2506, 21290, seed])
    Ls = np.array([W.box_length(int(M)) for M in sizes])
    xyz = np.concatenate([_start(int(M), L, rng) for M, L in zip(sizes, Ls)])
    types = np.tile(np.array([0, 1, 2], dtype=np.int32), int(np.sum(sizes)))
    one = len(sizes) == 1
    h = F.Handle(float(Ls[0]) if one else Ls, xyz, types, W.PAPER_POT, precision="fp32",
                 n_mol=None if one else np.asarray(sizes, dtype=np.int32))
    h.sweep(n_eq, T, W.PAPER_MIX, seed if one else np.arange(len(sizes), dtype=np.uint64) + np.uint64(seed))
    if precision != "fp32" or recompute:
        xyz, types, _ = h.state()
        h.close()
        h = F.Handle(float(Ls[0]) if one else Ls, xyz, types, W.PAPER_POT, precision=precision,
                     n_mol=None if one else np.asarray(sizes, dtype=np.int32), recompute_every=recompute)
    return h, Ls


def _qvectors(L, q0, n):
    """n wavevectors of the box near modulus q0."""
    return W.qvectors(L, q0, dq=0.6, max_n=n)


def _sizes(case):
    if case["R"] == 1 or case.get("M_hi", case["M"]) == case["M"]:
        return np.full(case["R"], case["M"])
    return W.replica_mix(case["R"], 0, case["M"], case["M_hi"])[0]


def prepare(case, seed):
    kind = case["kind"]
    s = {"kind": kind, "case": case, "seed": seed}
    if kind in ("sweep", "restart"):
        sizes = _sizes(case)
        R = len(sizes)
        T = case["T"] if R == 1 else np.random.default_rng([8, seed]).uniform(case["T"], max(case["T"], W.T_HIGH), size=R)
        big = int(np.sum(sizes)) > 20000
        s["h"], _ = _system(sizes, T, seed, case["precision"], case["recompute"], 100 if big else 400)
        s["T"], s["mix"] = T, MIXES[case["mix"]]
        s["seeds"] = seed + 17 if R == 1 else np.arange(R, dtype=np.uint64) + np.uint64(seed + 17)
        if case["tune"]:
            s["h"].autotune(case["tune"], T, s["mix"], s["seeds"])
        if kind == "restart":
            s["xyz"], s["types"], _ = s["h"].state()
    elif kind == "corr":
        R = case["R"]
        s["h"], Ls = _system(np.full(R, case["M"]), case["T"], seed)
        s["qa"], s["qc"] = _qvectors(Ls[0], 7.4, case["n_q"]), _qvectors(Ls[0], 5.1, case["n_q"])
        s["T"], s["mix"] = np.full(R, case["T"]), MIXES[case["mix"]]
        s["seeds"] = np.arange(R, dtype=np.uint64) + np.uint64(seed + 17)
        s["lags"], s["every"] = SP.log_lags(case["lag_max"]), max(1, case["lag_max"] // 8)
        s["h"].corr_setup(s["lags"], s["every"], case["origins"], s["qa"], s["qc"])
    elif kind == "obs":
        s["h"], Ls = _system(np.full(case["R"], case["M"]), case["T"], seed)
        s["Ls"] = Ls
        s["qa"], s["qc"] = _qvectors(Ls[0], 7.4, case["n_q"]), _qvectors(Ls[0], 5.1, case["n_q"])
        s["q0"], s["X0"], s["t0"] = s["h"].state_fixed()
        s["h"].set_t0()
        s["h"].sweep(case["sweeps"], case["T"], W.PAPER_MIX, seed + 17)
    elif kind == "static":
        s["h"], Ls = _system(np.full(case["R"], case["M"]), case["T"], seed)
        s["Ls"] = Ls
        s["q"] = np.concatenate([_qvectors(Ls[0], q0, case["n_q"] // 3) for q0 in (2.0, 5.1, 7.4)])
        s["dr"] = 0.5 * Ls[0] / case["bins"] * (1.0 - 1e-9)
        s["T"] = case["T"]
    elif kind == "md":
        s["h"], Ls = _system([case["M"]], case["T"], seed, n_eq=200 if case["M"] > 20000 else 600)
        s["L"] = Ls[0]
        s["v0"] = W.maxwell_velocities(3 * case["M"], case["T"], seed)
        s["h"].md_setup(0.001, case["tau"], case["T"], s["v0"], case["forces"])
    else:
        raise ValueError("unknown kind %r" % kind)
    return s


def run(s):
    kind, c, h = s["kind"], s["case"], s["h"]
    if kind in ("sweep", "restart"):
        if kind == "restart":
            h.set_state(s["xyz"], s["types"])
        h.sweep(c["sweeps"], s["T"], s["mix"], s["seeds"])
        E = h.energy()
        xyz, types, st = h.state()
        counts = np.array([x["attempts"] + x["accepts"] + [x[k] for k in STATS] for x in st], dtype=np.int64)
        return {"E": E, "xyz": xyz, "types": types, "counts": counts}
    if kind == "corr":
        h.corr_run(c["sweeps"], s["T"], s["mix"], s["seeds"])
        return {"sums": h.corr_sums(), "results": h.corr_results(), "tau": h.corr_relaxation_time(0)}
    if kind == "obs":
        out, fs, fcm, c2 = h.observables(s["qa"], s["qc"], per_particle=True)
        return {"out": out, "fs": fs, "fcm": fcm, "c2": c2}
    if kind == "static":
        S = h.structure_factor(s["q"])
        counts, g = h.pair_histogram(s["dr"], c["bins"])
        return {"S": S, "counts": counts.astype(np.int64), "g": g, "P": h.pressure(s["T"]), "E": h.energy()}
    h.md_run(c["steps"])
    v, out = h.md_state()
    xyz, types, _ = h.state()
    return {"v": v, "out": out, "xyz": xyz}


# --- what a pass cannot do without -----------------------------------------------------------------------------------


def _mean_M(case):
    return 0.5 * (case["M"] + case.get("M_hi", case["M"]))


def _neighbourhood(M):
    """Atoms in the 27 cells around a cell (the cells are at least 1.575 wide)."""
    L, nc = W.box_length(M), 2
    while L / (nc + 2) >= 1.575:
        nc += 2
    return 3.0 * M * min(1.0, 27.0 / nc ** 3)


def work(case):
    kind, M = case["kind"], _mean_M(case)
    N = 3.0 * M * case.get("R", 1)
    if kind in ("sweep", "restart"):
        # old and new distance of every neighbour (8 flops each), 19 pair terms in range (10 each); about a fifth of the
        # attempts is refused before any distance.  State in and out, with its types, and the energies.
        flops = N * case["sweeps"] * 0.8 * (16.0 * _neighbourhood(M) + 190.0)
        return {"bytes": N * (16 + 28) + (28 * N if kind == "restart" else 0), "flops": flops}
    if kind == "corr":
        lags = SP.log_lags(case["lag_max"])
        n = case["sweeps"] * min(1.0 / max(1, case["lag_max"] // 8), case["origins"] / float(case["lag_max"]))
        pairs = max(1.0, n * len(lags))
        attempts = N * case["sweeps"] * 0.8 * (16.0 * _neighbourhood(M) + 190.0)
        return {"bytes": N * (16 + 24) + pairs * 1000.0, "flops": attempts + pairs * (N + N / 3) * case["n_q"] * 30.0}
    if kind == "obs":
        return {"bytes": N * (16 + 24 + 8 + 28 / 3 + 16 / 3), "flops": (N + N / 3) * case["n_q"] * 30.0}
    if kind == "static":
        n = 3.0 * M
        flops = case["R"] * (n * (n - 1) / 2 * 10.0 + n * (case["n_q"] // 3 * 3) * 50.0 + n * 12.0 * 60.0)
        return {"bytes": N * 16 + case["R"] * (case["bins"] * 16 + case["n_q"] * 8), "flops": flops}
    # md: about 5 pairs in range per atom and step, 40 flops each, found among half the neighbours (10 flops each)
    return {"bytes": N * (16 + 24 + 48), "flops": N * case["steps"] * (5 * 40.0 + 0.5 * 10.0 * _neighbourhood(M))}


# --- the same in 64 bits, with torch and numpy -----------------------------------------------------------------------

_TWO32 = 4294967296.0


def _dev():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _int_pos(q):
    return torch.from_numpy(np.ascontiguousarray(np.asarray(q, dtype=np.uint32)).view(np.int32)).to(_dev())


def _pairs(qi, L, r):
    """All pairs i < j closer than r (qi: int32 positions, whose wrapping differences are the minimum image)."""
    n, h = qi.shape[0], np.float32(L / _TWO32)
    step = max(1, (1 << 26) // n)
    found = []
    for a in range(0, n, step):
        d2 = 0.0
        for ax in range(3):
            d = (qi[None, a:, ax] - qi[a:a + step, None, ax]).to(torch.float32) * float(h)
            d2 = d2 + d * d
        i, j = torch.nonzero(d2 < r * r, as_tuple=True)
        keep = j > i
        found.append(torch.stack([i[keep] + a, j[keep] + a]))
    return torch.cat(found, dim=1)


def _pair_terms(qi, types, L, ij):
    """(energy, -r dphi/dr, separation, r^2) of each pair: WCA inside its cutoff, FENE inside a molecule."""
    sig = torch.tensor(W.SIGMA, dtype=torch.float64, device=qi.device)
    i, j = ij
    d = (qi[j] - qi[i]).to(torch.float64) * (float(L) / _TWO32)
    r2 = (d * d).sum(dim=1)
    sab = 0.5 * (sig[types[i]] + sig[types[j]])
    s6 = (sab * sab / r2) ** 3
    inside = r2 < 2.0 ** (1.0 / 3.0) * sab * sab
    zero = torch.zeros_like(r2)
    u = torch.where(inside, 4.0 * W.EPS * (s6 * s6 - s6) + W.EPS, zero)
    w = torch.where(inside, 24.0 * W.EPS * s6 * (2.0 * s6 - 1.0), zero)
    bonded = torch.div(i, 3, rounding_mode="floor") == torch.div(j, 3, rounding_mode="floor")
    x = torch.where(bonded, r2 / (W.FENE_R0 * sab) ** 2, zero)
    u = u - W.FENE_K * W.EPS * torch.log1p(-x)
    w = w - 2.0 * W.FENE_K * W.EPS * x / (1.0 - x)
    return u, w, d, r2


_REACH = 1.66  # longer than every cutoff (1.235) and every bond (1.575)


def _exact_static(s):
    h, c = s["h"], s["case"]
    q, _, t = h.state_fixed()
    n, R, L = 3 * c["M"], c["R"], float(s["Ls"][0])
    S, counts, P, E = [], [], [], []
    for r in range(R):
        qr, tr = q[r * n:(r + 1) * n], torch.from_numpy(t[r * n:(r + 1) * n].astype(np.int64)).to(_dev())
        x = torch.from_numpy(qr.astype(np.float64) * (L / _TWO32)).to(_dev())
        ph = x @ torch.from_numpy(s["q"]).to(_dev()).T
        S.append(((torch.cos(ph).sum(dim=0) ** 2 + torch.sin(ph).sum(dim=0) ** 2) / n).cpu().numpy())
        qi = _int_pos(qr)
        hist = torch.zeros(c["bins"], dtype=torch.int64, device=_dev())
        step = max(1, (1 << 25) // n)
        for a in range(0, n, step):
            r2 = 0.0
            for ax in range(3):
                d = (qi[None, a:, ax] - qi[a:a + step, None, ax]).to(torch.float64) * (L / _TWO32)
                r2 = r2 + d * d
            later = torch.arange(r2.shape[1], device=_dev())[None, :] > torch.arange(r2.shape[0], device=_dev())[:, None]
            b = torch.floor(torch.sqrt(r2[later]) / s["dr"]).to(torch.int64)
            hist += torch.bincount(b[b < c["bins"]], minlength=c["bins"])
        counts.append(hist.cpu().numpy())
        u, w, _, _ = _pair_terms(qi, tr, L, _pairs(qi, L, _REACH))
        E.append(float(u.sum()))
        P.append([float(w.sum()), n * s["T"] / L ** 3 + float(w.sum()) / (3.0 * L ** 3)])
    counts = np.array(counts)
    edge = np.arange(c["bins"] + 1) * s["dr"]
    shell = 4.0 / 3.0 * math.pi * (edge[1:] ** 3 - edge[:-1] ** 3)
    g = 2.0 * counts / (n * (n / L ** 3) * shell)
    return {"S": np.array(S), "counts": None, "g": g, "P": np.array(P), "E": np.array(E)}


def _orientation(q, L, ref):
    q3 = q.reshape(-1, 3, 3)
    rel = (q3 - q3[:, :1]).view(np.int32).astype(np.float64) * (L / _TWO32)
    u = rel[np.arange(len(rel)), ref] - rel.mean(axis=1)
    return u / np.linalg.norm(u, axis=1, keepdims=True)


def _relax(L, q, X, q0, X0, t0, qa, qc):
    """Per particle F_s (atoms), F_s^cm and C_2 (molecules)."""
    isB = t0.reshape(-1, 3) == 1
    ref = np.where(isB.any(axis=1), np.argmax(isB, axis=1), 0)
    d = torch.from_numpy((X - X0).astype(np.float64) * (L / _TWO32)).to(_dev())
    fs = torch.cos(d @ torch.from_numpy(qa).to(_dev()).T).mean(dim=1).cpu().numpy()
    cm = d.reshape(-1, 3, 3).sum(dim=1) / 3.0
    fcm = torch.cos(cm @ torch.from_numpy(qc).to(_dev()).T).mean(dim=1).cpu().numpy()
    x = (_orientation(q, L, ref) * _orientation(q0, L, ref)).sum(axis=1)
    return fs, fcm, 1.5 * x * x - 0.5


def _exact_obs(s):
    c, n = s["case"], 3 * s["case"]["M"]
    q, X, _ = s["h"].state_fixed()
    got = [_relax(float(L), *(a[r * n:(r + 1) * n] for a in (q, X, s["q0"], s["X0"], s["t0"])), s["qa"], s["qc"])
           for r, L in enumerate(s["Ls"])]
    return {"out": np.array([[x.mean() for x in g] for g in got]), "fs": np.concatenate([g[0] for g in got]),
            "fcm": np.concatenate([g[1] for g in got]), "c2": np.concatenate([g[2] for g in got])}


def _exact_corr(s):
    """The sums over the states that the same sweeps, made one at a time, pass through."""
    c, h = s["case"], s["h"]
    R, n, L = c["R"], 3 * c["M"], W.box_length(c["M"])
    lags = [int(x) for x in s["lags"]]
    sums = np.zeros((R, len(lags), F.MC_CORR_NSUM))
    live = []

    def sample(o, l, now):
        for r in range(R):
            k = slice(r * n, (r + 1) * n)
            fs, fcm, c2 = _relax(L, now[0][k], now[1][k], o[1][0][k], o[1][1][k], o[1][2][k], s["qa"], s["qc"])
            sums[r, l, :14] += [1, fs.mean(), fs.mean() ** 2, fs.sum(), (fs * fs).sum(), fcm.mean(), fcm.mean() ** 2, fcm.sum(),
                                (fcm * fcm).sum(), c2.mean(), c2.mean() ** 2, c2.sum(), (c2 * c2).sum(), (c2 * fcm).sum()]

    for t in range(c["sweeps"] + 1):
        if t:
            h.sweep(1, s["T"], s["mix"], s["seeds"])
        due = [(o, lags.index(t - o[0])) for o in live if t - o[0] in lags]
        fresh = t % s["every"] == 0
        now = h.state_fixed() if due or fresh else None
        for o, l in due:
            sample(o, l, now)
        live = [o for o in live if t - o[0] < lags[-1]]
        if fresh and len(live) < c["origins"]:
            live.append((t, now))
            if lags[0] == 0:
                sample(live[-1], 0, now)
    return {"sums": sums, "results": None, "tau": None}


def _exact_md(s):
    c, L, dt = s["case"], float(s["L"]), 0.001
    q, _, t = s["h"].state_fixed()
    dev = _dev()
    types = torch.from_numpy(t.astype(np.int64)).to(dev)
    qi = _int_pos(q)
    v = torch.from_numpy(s["v0"]).to(dev)
    n, T = v.shape[0], c["T"]
    g, per = 3.0 * n, dt * (_TWO32 / L)
    Q = g * T * c["tau"] ** 2 if c["tau"] > 0 else None
    xi = eta = 0.0

    def forces(ij):
        u, w, d, r2 = _pair_terms(qi, types, L, ij)
        f = (w / r2)[:, None] * d
        return torch.zeros_like(v).index_add_(0, ij[1], f).index_add_(0, ij[0], -f), float(u.sum())

    ij = _pairs(qi, L, _REACH + 0.35)
    f, U = forces(ij)
    for k in range(c["steps"]):
        if Q:
            xi += 0.5 * dt * (float((v * v).sum()) - g * T) / Q
            eta += 0.5 * dt * xi
        v = v * math.exp(-xi * 0.5 * dt) + 0.5 * dt * f
        step = torch.round(v * per).to(torch.int64)
        qi = ((qi.to(torch.int64) + step + (1 << 31)) % (1 << 32) - (1 << 31)).to(torch.int32)
        if k % 20 == 19:
            ij = _pairs(qi, L, _REACH + 0.35)
        f, U = forces(ij)
        v = (v + 0.5 * dt * f) * math.exp(-xi * 0.5 * dt)
        if Q:
            xi += 0.5 * dt * (float((v * v).sum()) - g * T) / Q
            eta += 0.5 * dt * xi
    K = 0.5 * float((v * v).sum())
    xyz = (qi.to(torch.int64) % (1 << 32)).to(torch.float64) * (L / _TWO32)
    bath = 0.5 * Q * xi * xi + g * T * eta if Q else 0.0
    return {"v": v.cpu().numpy(), "out": np.array([[K, U, xi, eta, K + U + bath]]), "xyz": xyz.cpu().numpy()}


def exact(case, seed):
    kind = case["kind"]
    if kind in ("sweep", "restart"):
        return None  # where a chain of accepted and refused moves ends has no value of its own
    s = prepare(case, seed)  # the inputs; what is returned is computed here
    if kind == "md":
        return _exact_md(s)
    return {"corr": _exact_corr, "obs": _exact_obs, "static": _exact_static}[kind](s)
