"""The work a user has this library do, as cases that can be timed.

Each case is one call chain of the public Python binding
(``paper_1006_0252_gb300.pa``), with sizes from the workloads of
``inputs.py``, the benchmark and the tests.  ``prepare`` holds what a program
keeps between annealing runs (the ``Run``, ``Batch`` or ``Server`` and its
buffers); ``run`` is one complete use of it, from a fresh beta = 0 population
to the results on the host; ``exact`` restates the +-1 cubic run and the
averages of Sec. 3 in numpy, without this library.
"""
from __future__ import annotations

import math

import numpy as np

from paper_1006_0252_gb300 import inputs, pa

# Integer operations per attempted flip: a quarter of a Philox4x32-10 block
# (10 rounds x 4 operations / 4 sites), one compare, one decision.
OPS_PER_FLIP = 12


def listed() -> list[dict]:
    return [
        # A program that watches the run: one step, read the observables, decide
        # on the next beta.  The smallest calls: launches and latency count.
        {"name": "steps_l4", "kind": "steps", "L": 4, "R0": 1000, "steps": 10, "beta_max": 1.0, "theta": 10},
        # The small workload (3D L=4, R0=1000, 101 betas), whole schedule.
        {"name": "run_l4", "kind": "run", "L": 4, "R0": 1000, "steps": 100, "beta_max": 5.0, "theta": 10},
        # The benchmark workload: 3D L=8, R0=1e5, 201 betas, whole schedule.
        {"name": "run_l8", "kind": "run", "L": 8, "R0": 100_000, "steps": 200, "beta_max": 5.0, "theta": 10},
        # The largest edge of the serving mix at an odd population.
        {"name": "run_l12", "kind": "run", "L": 12, "R0": 30_011, "steps": 51, "beta_max": 5.0, "theta": 10},
        # Many runs of uneven L and R0 in one graph, with the Sec. 3 estimators
        # and the overlap of pairs of runs (the batched workload, fewer runs).
        {"name": "batch_mixed", "kind": "batch", "realisations": 6, "runs": 4, "L_lo": 6, "L_hi": 10,
         "R_lo": 20_000, "R_hi": 80_000, "mix": 3, "steps": 25, "beta_max": 5.0, "theta": 10},
        # The open +-1 chain N=4096 at R0=2e5, theta=5, fewer temperatures.
        {"name": "chain_4096", "kind": "chain", "N": 4096, "R0": 200_000, "steps": 40, "beta_max": 4.0, "theta": 5,
         "periodic": False},
        # The paper's 3D study (Gaussian couplings, L=8, R=2000, theta=100, 50
        # runs a realisation), fewer realisations and temperatures, with its
        # estimators, their bootstrap errors and the overlap.
        {"name": "gauss_set_3d", "kind": "gauss_set", "dim": 3, "L": 8, "realisations": 4, "runs": 50, "R0": 2000,
         "steps": 15, "theta": 100, "B": 100},
        # The paper's 1D study (periodic Gaussian chain, N=256, R=1000, theta=50).
        {"name": "gauss_set_1d", "kind": "gauss_set", "dim": 1, "L": 256, "realisations": 4, "runs": 50, "R0": 1000,
         "steps": 25, "theta": 50, "B": 100},
        # One Gaussian run beyond the paper's size.
        {"name": "gauss_l10", "kind": "gauss_run", "L": 10, "R0": 20_000, "steps": 40, "beta_max": 4.0, "theta": 10},
        # Requests of different sizes through the continuous-batching server.
        {"name": "serve", "kind": "serve", "requests": 8, "R_lo": 10_000, "R_hi": 60_000, "steps_lo": 51,
         "steps_hi": 101, "mix": 5, "theta": 10},
        # A box with open z faces (slab geometry), which takes the general kernel.
        {"name": "box_slab", "kind": "box", "Lx": 8, "Ly": 6, "Lz": 5, "mask": 3, "gaussian": False, "R0": 20_000,
         "steps": 20, "beta_max": 3.0, "theta": 10},
        # Sec. 3 on finished runs: weighted average, its bootstrap error and the
        # pair-weighted average, host arrays in, numbers out.
        {"name": "averages", "kind": "averages", "M": 200, "B": 1000},
    ]


def _log(rng, lo: float, hi: float) -> int:
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _steps_for(rng, lo: int, hi: int, flips_per_step: float, most: float) -> int:
    """A number of steps in [lo, hi] whose flips stay below `most`."""
    return max(1, min(_log(rng, lo, hi), int(most / flips_per_step)))


def draw(rng) -> dict:
    kind = rng.choice(["steps", "run", "run", "run", "batch", "chain", "gauss_set", "gauss_run", "serve", "box",
                       "averages"])
    if kind == "steps":
        return {"kind": kind, "L": rng.choice([4, 6]), "R0": _log(rng, 300, 3000), "steps": rng.randint(4, 16),
                "beta_max": round(rng.uniform(0.5, 2.0), 3), "theta": rng.randint(1, 12)}
    if kind == "run":
        L = rng.choice([2, 4, 6, 8, 10, 12, 14, 16])
        R0 = _log(rng, 1000, 200_000)
        theta = rng.choice([5, 10, 10, 20])
        if R0 * L ** 3 * theta * 20 > 1.0e11:
            R0 = int(1.0e11 / (L ** 3 * theta * 20))
        return {"kind": kind, "L": L, "R0": R0, "steps": _steps_for(rng, 20, 200, R0 * L ** 3 * theta, 1.0e11),
                "beta_max": round(rng.uniform(1.0, 5.0), 3), "theta": theta}
    if kind == "batch":
        lo, hi = rng.choice([(4, 8), (6, 10), (6, 10), (8, 12)])
        return {"kind": kind, "realisations": rng.randint(2, 6), "runs": rng.randint(2, 5), "L_lo": lo, "L_hi": hi,
                "R_lo": _log(rng, 1000, 20_000), "R_hi": _log(rng, 20_001, 50_000), "mix": rng.randint(1, 1000),
                "steps": rng.randint(8, 20), "beta_max": round(rng.uniform(1.0, 5.0), 3), "theta": 10}
    if kind == "chain":
        periodic = rng.random() < 0.3
        N = _log(rng, 64, 4096)
        N = N // 2 * 2 if periodic else N
        R0 = _log(rng, 1000, 200_000)
        theta = rng.choice([5, 10])
        return {"kind": kind, "N": N, "R0": R0, "steps": _steps_for(rng, 20, 100, R0 * N * theta, 1.5e11),
                "beta_max": round(rng.uniform(1.0, 4.0), 3), "theta": theta, "periodic": periodic}
    if kind == "gauss_set":
        dim = rng.choice([1, 3])
        L = rng.choice([4, 6, 8]) if dim == 3 else _log(rng, 32, 256) * 2
        return {"kind": kind, "dim": dim, "L": L, "realisations": rng.randint(1, 4), "runs": rng.randint(8, 50),
                "R0": _log(rng, 500, 2500), "steps": rng.randint(5, 15), "theta": rng.choice([25, 50]),
                "B": rng.choice([50, 100])}
    if kind == "gauss_run":
        L = rng.choice([4, 6, 8, 8, 10, 12])
        R0 = _log(rng, 1000, 100_000)
        if R0 * L ** 3 * 10 * 10 > 4.0e10:
            R0 = int(4.0e10 / (L ** 3 * 10 * 10))
        return {"kind": kind, "L": L, "R0": R0, "steps": _steps_for(rng, 10, 80, R0 * L ** 3 * 10, 4.0e10),
                "beta_max": round(rng.uniform(1.0, 4.0), 3), "theta": 10}
    if kind == "serve":
        return {"kind": kind, "requests": rng.randint(3, 8), "R_lo": 10_000, "R_hi": _log(rng, 20_000, 60_000),
                "steps_lo": 51, "steps_hi": rng.randint(60, 101), "mix": rng.randint(1, 1000), "theta": 10}
    if kind == "box":
        return {"kind": kind, "Lx": rng.choice([4, 6, 8]), "Ly": rng.choice([4, 6, 8]), "Lz": rng.randint(3, 8),
                "mask": 3, "gaussian": rng.random() < 0.4, "R0": _log(rng, 1000, 30_000), "steps": rng.randint(5, 20),
                "beta_max": round(rng.uniform(0.5, 3.0), 3), "theta": rng.choice([5, 10])}
    return {"kind": "averages", "M": _log(rng, 8, 2000), "B": _log(rng, 50, 2000)}


# ---- sizes a case fixes by itself (the seed only makes couplings and random numbers) ------------


def _betas(case: dict) -> np.ndarray:
    return inputs.linear_schedule(case["beta_max"], case["steps"] + 1)[1:]


def _gauss_set_betas(case: dict) -> np.ndarray:
    """`steps` temperatures of the paper's own schedule, evenly thinned."""
    full = inputs.paper_schedule_3d() if case["dim"] == 3 else inputs.paper_schedule_1d()
    at = np.rint(np.linspace(0, len(full) - 1, case["steps"] + 1)).astype(int)[1:]
    return full[at]


def _batch_sizes(case: dict) -> list[tuple[int, int]]:
    """(L, R0) of every run, realisation by realisation."""
    Ls = list(range(case["L_lo"], case["L_hi"] + 1, 2))
    R = inputs.uniform_ints(case["realisations"] * case["runs"], case["R_lo"], case["R_hi"], seed=case["mix"])
    return [(Ls[d % len(Ls)], int(R[d * case["runs"] + r])) for d in range(case["realisations"])
            for r in range(case["runs"])]


def _requests(case: dict) -> list[tuple[int, int, int]]:
    """(L, R0, steps) of every request."""
    q = inputs.serving_requests(case["requests"], seed=case["mix"], r_lo=case["R_lo"], r_hi=case["R_hi"],
                                steps_lo=case["steps_lo"], steps_hi=case["steps_hi"], theta=case["theta"])
    return [(r.spec.L, r.spec.R0, len(r.spec.betas) - 1) for r in q]


def _averages_inputs(case: dict, seed: int):
    """-beta F~ of M runs (the paper's Var(-beta F~) of a few tenths), their
    energies and population targets."""
    rng = np.random.default_rng(seed)
    M = case["M"]
    x = 1147.8 + math.sqrt(0.34) * rng.standard_normal(M)
    A = -224.2 + 0.5 * rng.standard_normal(M)
    R = np.where(rng.random(M) < 0.5, 1000.0, 3000.0)
    return x, A, R


# ---- one case ------------------------------------------------------------------------------------


def prepare(case: dict, seed: int) -> dict:
    """The handle a program keeps and the host arrays it calls it with."""
    kind = case["kind"]
    s: dict = {"case": case, "seed": seed}
    if kind in ("steps", "run"):
        J = inputs.couplings_3d(case["L"], 0, seed)
        s["run"] = pa.Run(J, case["L"], 3, case["R0"], seed)
        s["betas"] = _betas(case)
    elif kind == "chain":
        J = inputs.couplings_chain(case["N"], 0, seed, open_chain=not case["periodic"])
        s["run"] = pa.Run(J, case["N"], 1, case["R0"], seed)
        s["betas"] = _betas(case)
    elif kind == "gauss_run":
        J = inputs.gaussian_couplings_3d(case["L"], 0, seed)
        s["run"] = pa.Run(J, case["L"], 3, case["R0"], seed, gaussian=True)
        s["betas"] = _betas(case)
    elif kind == "box":
        Ls = (case["Lx"], case["Ly"], case["Lz"])
        make = inputs.gaussian_couplings_lattice if case["gaussian"] else inputs.couplings_lattice
        s["run"] = pa.Run(make(*Ls, 0, seed), 0, 3, case["R0"], seed, gaussian=case["gaussian"], Ls=Ls,
                          periodic_mask=case["mask"])
        s["betas"] = _betas(case)
    elif kind == "batch":
        b = _betas(case)
        specs = [inputs.RunSpec(3, L, i // case["runs"], seed + i, R0, b, case["theta"], coupling_seed=seed)
                 for i, (L, R0) in enumerate(_batch_sizes(case))]
        s["batch"] = pa.Batch(specs)
        s["betas"] = b
        # pairs of runs of one realisation
        n = case["runs"]
        s["a"] = np.array([d * n for d in range(case["realisations"])], dtype=np.int32)
        s["b"] = s["a"] + 1
    elif kind == "gauss_set":
        b = _gauss_set_betas(case)
        n = case["runs"]
        specs = [inputs.RunSpec(case["dim"], case["L"], d, seed + (d << 8 | r), case["R0"], b, case["theta"],
                                coupling_seed=seed, gaussian=True, open_chain=False)
                 for d in range(case["realisations"]) for r in range(n)]
        s["batch"] = pa.Batch(specs)
        s["betas"] = b
        a = np.concatenate([d * n + np.arange(n // 2) for d in range(case["realisations"])]).astype(np.int32)
        s["a"], s["b"] = a, a + n // 2
    elif kind == "serve":
        s["server"] = pa.Server(max_runs=256)
        s["requests"] = [(L, inputs.couplings_3d(L, i, seed), R0, seed + i, inputs.linear_schedule(5.0, n + 1)[1:])
                         for i, (L, R0, n) in enumerate(_requests(case))]
    else:
        s["x"], s["A"], s["R"] = _averages_inputs(case, seed)
        s["x2"], s["A2"], s["R2"] = _averages_inputs(case, seed + 1)
    return s


def _population(s: dict) -> dict:
    """The final population in buffers of the run's capacity that the program
    keeps (slots past the population size stay zero): the energies, and the
    spins where a program would look at all of them."""
    r, cap = s["run"], inputs.default_capacity(s["case"]["R0"])
    E = r.energies()
    if "energies" not in s:
        s["energies"] = np.zeros(cap, dtype=np.int32)
        s["spins"] = np.zeros((cap, r.N), dtype=np.int8) if cap * r.N <= 8_000_000 else None
    s["energies"][:len(E)] = E
    out = {"energies": s["energies"]}
    if s["spins"] is not None:
        s["spins"][:len(E)] = r.spins()
        out["spins"] = s["spins"]
    return out


def run(s: dict):
    case, kind = s["case"], s["case"]["kind"]
    if kind == "steps":
        r, rows = s["run"], []
        r.reset(s["seed"])
        for beta in s["betas"]:
            r.step(float(beta), case["theta"])
            rows.append(r.observables())
        out = {k: np.array([o[k] for o in rows]) for k in ("E_mean", "E2_mean", "minus_beta_F", "lnQ_last", "R")}
        return out | _population(s)
    if kind in ("run", "chain", "gauss_run", "box"):
        r = s["run"]
        r.reset(s["seed"])
        r.run_schedule(s["betas"], case["theta"])
        out = dict(r.trajectory(len(s["betas"]) + 1))
        if kind == "gauss_run" or (kind == "box" and case["gaussian"]):
            out |= r.trajectory_energy(len(s["betas"]) + 1)
        return out | _population(s)
    if kind == "batch":
        b, n = s["batch"], len(s["betas"]) + 1
        b.reset()
        b.run(s["betas"], case["theta"])
        out = dict(b.trajectory(n))
        out |= b.diagnostics(case["runs"], n)
        out["gamma"], out["pairs"] = b.overlap(s["a"], s["b"])
        return out
    if kind == "gauss_set":
        b, n = s["batch"], len(s["betas"]) + 1
        b.reset()
        b.run(s["betas"], case["theta"])
        out = {"results_" + k: v for k, v in b.results().items()}
        out |= b.energy(n)
        out |= b.diagnostics(case["runs"], n)
        out |= b.bootstrap(case["runs"], n, case["B"])
        out["gamma"], out["pairs"] = b.overlap(s["a"], s["b"])
        out["hist"] = b.overlap_hist(s["a"], s["b"])
        return out
    if kind == "serve":
        srv = s["server"]
        ids = [srv.submit(3, L, J, R0, seed, betas, case["theta"]) for L, J, R0, seed, betas in s["requests"]]
        done = 0
        while done < len(ids):
            done += srv.tick(2)[2]
        res = [srv.result(i, len(q[4]) + 1) for i, q in zip(ids, s["requests"])]
        out = {k: np.array([r[k] for r in res]) for k in ("status", "R", "minus_beta_F", "E_mean", "sumE", "sumE2",
                                                          "flips")}
        out["trajectory"] = [r["trajectory"] for r in res]
        return out
    mean, fbar = pa.pa_weighted_average(s["x"], s["A"], s["R"])
    sd_mean, sd_fbar = pa.pa_bootstrap(s["x"], s["A"], s["R"], case["B"], s["seed"])
    pair_mean, pair_fbar = pa.pa_weighted_average_pairs(s["x"], s["x2"], s["A"], s["R"], s["R2"])
    return {"mean": mean, "fbar": fbar, "sd_mean": sd_mean, "sd_fbar": sd_fbar, "pair_mean": pair_mean,
            "pair_fbar": pair_fbar}


def work(case: dict) -> dict:
    """Couplings in, results out; the integer operations of the attempted
    flips, or the exponentials and sums of the averages."""
    kind = case["kind"]
    if kind in ("steps", "run"):
        N, R, st, th = case["L"] ** 3, case["R0"], case["steps"], case["theta"]
        runs, coup = [(N, R, st, th)], 3 * N
    elif kind == "chain":
        runs, coup = [(case["N"], case["R0"], case["steps"], case["theta"])], case["N"]
    elif kind == "gauss_run":
        N = case["L"] ** 3
        runs, coup = [(N, case["R0"], case["steps"], case["theta"])], 12 * N
    elif kind == "box":
        N = case["Lx"] * case["Ly"] * case["Lz"]
        runs, coup = [(N, case["R0"], case["steps"], case["theta"])], 3 * N * (4 if case["gaussian"] else 1)
    elif kind == "batch":
        runs = [(L ** 3, R, case["steps"], case["theta"]) for L, R in _batch_sizes(case)]
        coup = sum(3 * r[0] for r in runs)
    elif kind == "gauss_set":
        N = case["L"] ** 3 if case["dim"] == 3 else case["L"]
        runs = [(N, case["R0"], case["steps"], case["theta"])] * (case["realisations"] * case["runs"])
        coup = 4 * (3 if case["dim"] == 3 else 1) * N * len(runs)
    elif kind == "serve":
        runs = [(L ** 3, R, n, case["theta"]) for L, R, n in _requests(case)]
        coup = sum(3 * r[0] for r in runs)
    else:
        M, B = case["M"], case["B"]
        return {"bytes": 8.0 * (5 * M + 6), "flops": 20.0 * M * (B + 4)}
    # the final population (packed spins and energies) and the per-step record
    out = sum(R * (N / 8 + 4) + 48 * (st + 1) for N, R, st, _ in runs)
    return {"bytes": float(coup + out), "flops": float(OPS_PER_FLIP * sum(N * R * st * th for N, R, st, th in runs))}


# ---- the same in 64 bits ---------------------------------------------------------------------------
# Numpy restatements: the annealing run of a periodic +-1 cubic lattice
# (Sec. 2) with its random numbers (Philox4x32-10, counters as documented in
# the library's numerics specification), and the estimators of Sec. 3.

_M0, _M1 = np.uint64(0xD2511F53), np.uint64(0xCD9E8D57)
_U32 = np.uint64(0xFFFFFFFF)
_S32 = np.uint64(32)
_INIT, _RESAMPLE, _SWEEP, _BOOT = 0x1A000000, 0x2B000000, 0x3C000000, 0x4D000000


def _philox(seed: int, c0, c1, c2, c3):
    """The four 32-bit outputs (uint64 arrays) for counters (c0, c1, c2, c3)."""
    c0, c1, c2, c3 = (np.asarray(c, dtype=np.uint64) for c in (c0, c1, c2, c3))
    k0, k1 = seed & 0xFFFFFFFF, (seed >> 32) & 0xFFFFFFFF
    for _ in range(10):
        p0, p1 = _M0 * c0, _M1 * c2
        c0, c1, c2, c3 = (p1 >> _S32) ^ c1 ^ np.uint64(k0), p1 & _U32, (p0 >> _S32) ^ c3 ^ np.uint64(k1), p0 & _U32
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    return c0, c1, c2, c3


def _anneal(case: dict, seed: int):
    """Observables of every step, energies and spins of the final population."""
    L, theta, R0 = case["L"], case["theta"], case["R0"]
    N = L ** 3
    J = inputs.couplings_3d(L, 0, seed).astype(np.int64)
    k = max(d for d in range(1, L + 1) if L % d == 0 and d * L <= 32)
    G, S = L // k, k * L // 2
    x, y, z = (a.reshape(-1) for a in np.meshgrid(np.arange(L), np.arange(L), np.arange(L), indexing="ij"))
    i = x + L * (y + L * z)
    order = np.argsort(i)
    x, y, z = x[order], y[order], z[order]
    w, p = y * G + z % G, (z // G) * L + x

    def at(x, y, z):
        return (x % L) + L * ((y % L) + L * (z % L))

    plus = [at(x + 1, y, z), at(x, y + 1, z), at(x, y, z + 1)]
    minus = [at(x - 1, y, z), at(x, y - 1, z), at(x, y, z - 1)]
    colour = (x + y + z) & 1
    sites = []
    for c in (0, 1):
        v = np.flatnonzero(colour == c)
        sites.append(v[np.argsort(w[v] * S + p[v] // 2)])  # by colour rank
    # beta = 0 population
    words = np.stack(_philox(seed, np.arange((L * G + 3) // 4)[None], np.arange(R0)[:, None], 0, _INIT), -1)
    words = words.reshape(R0, -1)
    s = 1 - 2 * ((words[:, w] >> p.astype(np.uint64)) & np.uint64(1)).astype(np.int64)

    def energy(s):
        return sum((s * s[:, plus[d]] * J[d]).sum(1) for d in range(3))

    E = energy(s)
    beta, mbF, T = 0.0, N * math.log(2.0), 0
    rec = [(beta, 0.0, mbF, R0, int(E.sum()), int((E * E).sum()))]
    for step, bn in enumerate(_betas(case)):
        db = float(bn) - beta
        wgt = np.exp(-db * (E - E.min()))
        Q = float(wgt.sum())
        lnQ = math.log(Q) - math.log(len(E)) - db * int(E.min())
        mbF += lnQ
        a = R0 * wgt / Q
        m = np.maximum(1, np.ceil(a / 32)).astype(np.int64)
        am = a / m
        copies = np.zeros(len(E), dtype=np.int64)
        for piece in range(int(m.max())):
            j = np.flatnonzero(m > piece)
            r = _philox(seed, piece, j, step, _RESAMPLE)
            u = (((r[0] << _S32) | r[1]) >> np.uint64(11)).astype(np.float64) * 2.0 ** -53
            n, P = 0, np.exp(-am[j])
            C = P.copy()
            live = u >= C
            while live.any() and n < 512:
                n += 1
                copies[j[live]] += 1
                P = P * am[j] / n
                C = C + P
                live &= u >= C
        s = s[np.repeat(np.arange(len(E)), copies)]
        R = len(s)
        thr = [min(2 ** 32 - 1, math.floor(math.exp(-float(bn) * 2 * d) * 2 ** 32)) for d in range(7)]
        thr = np.array([2 ** 32] + thr[1:], dtype=np.uint64)
        slot = np.arange(R)[:, None]
        for _ in range(theta):
            for c in (0, 1):
                v = sites[c]
                u = np.stack(_philox(seed, np.arange((len(v) + 3) // 4)[None], slot, T, _SWEEP + c), -1)
                u = u.reshape(R, -1)[:, :len(v)]
                h = sum(s[:, plus[d][v]] * J[d][v] + s[:, minus[d][v]] * J[d][minus[d][v]] for d in range(3))
                half = np.maximum(0, -s[:, v] * h)  # dE / 2 of a flip
                s[:, v] = np.where(u < thr[half], -s[:, v], s[:, v])
            T += 1
        E = energy(s)
        beta = float(bn)
        rec.append((beta, lnQ, mbF, R, int(E.sum()), int((E * E).sum())))
    return rec, E.astype(np.int32), s.astype(np.int8)


def _weighted(x, A, R):
    y = x + np.log(R)
    e = np.exp(y - y.max(-1, keepdims=True))
    mean = (e * A).sum(-1) / e.sum(-1)
    top = x.max(-1, keepdims=True)
    return mean, top[..., 0] + np.log(np.exp(x - top).mean(-1))


def exact(case: dict, seed: int):
    kind = case["kind"]
    if kind == "averages":
        x, A, R = _averages_inputs(case, seed)
        x2, _, R2 = _averages_inputs(case, seed + 1)
        M = case["M"]
        mean, fbar = _weighted(x, A, R)
        r = _philox(seed, np.arange(case["B"])[:, None], np.arange(M)[None], 0, _BOOT)[0]
        k = ((r * np.uint64(M)) >> _S32).astype(np.int64)
        bm, bf = _weighted(x[k], A[k], R[k])
        pm, pf = _weighted(x + x2, A, R * R2)
        return {"mean": float(mean), "fbar": float(fbar), "sd_mean": float(bm.std(ddof=1)),
                "sd_fbar": float(bf.std(ddof=1)), "pair_mean": float(pm), "pair_fbar": float(pf)}
    if kind not in ("steps", "run") or case["R0"] * case["L"] ** 3 * case["theta"] * case["steps"] > 1.2e8:
        return None  # a Monte Carlo run of that size takes numpy minutes
    rec, E, s = _anneal(case, seed)
    beta, lnQ, mbF, R, sE, sE2 = (np.array(v) for v in zip(*rec))
    cap, N = inputs.default_capacity(case["R0"]), case["L"] ** 3
    E, s = np.pad(E, (0, cap - len(E))), np.pad(s, ((0, cap - len(s)), (0, 0)))
    out = {"energies": E, "spins": s} if cap * N <= 8_000_000 else {"energies": E}
    if kind == "steps":
        return out | {"E_mean": (sE / R)[1:], "E2_mean": (sE2 / R)[1:], "minus_beta_F": mbF[1:], "lnQ_last": lnQ[1:],
                      "R": R[1:]}
    return out | {"beta": beta, "lnQ": lnQ, "minus_beta_F": mbF, "R": R, "sumE": sE, "sumE2": sE2}
