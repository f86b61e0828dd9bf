"""The work that users of the framework have it do, as cases that can be timed and compared.

Every case goes through the public Python binding (pa.Run, pa.Batch, pa.Server,
pa.resample_counts_noalloc): whole annealing runs from the smallest to the headline size, both
coupling models, fixed and adaptive schedules, one and two populations, lattices beyond a
shared-memory tile, many runs at once, and the calls that take a population out of the library
and back in.  Sizes are those of the repository's workloads, tests and benchmark, or lie between
them.
"""
from __future__ import annotations

import ctypes
import math
import random
from typing import List, Optional

import numpy as np
import torch

from paper_1711_02146_gb300 import pa
from paper_1711_02146_gb300.workloads import Workload, batched_mix, linear_betas, serving_stream

_ROWS = 1024  # rows of the observables of an adaptive run, whose number of steps depends on its energies


# ---------------------------------------------------------------- the cases

def listed() -> List[dict]:
    return [
        # the smallest call: a teaching- or test-sized run, every observable and the population read
        dict(name="small_run", kind="run", L=4, R=1000, n_temps=51, beta_max=5.0, n_sweeps=10, n_pop=1, eps=0.0,
             model=0, schedule="flat", spins=True),
        # P(q) of one sample: two populations on the same couplings, all temperatures' observables
        dict(name="overlap_run", kind="run", L=8, R=100_000, n_temps=201, beta_max=5.0, n_sweeps=10, n_pop=2,
             eps=0.0, model=0, schedule="flat", spins=False),
        # the headline: one large population annealed at a constant culling fraction, observables read as it goes
        dict(name="adaptive_large", kind="run", L=10, R=1_000_000, n_temps=4096, beta_max=5.0, n_sweeps=10, n_pop=1,
             eps=0.272, model=0, schedule="flat", spins=False),
        # the optimised schedule's sweeps (few at high and low temperature, many between), a population
        # that fills no whole number of tiles
        dict(name="scheduled_run", kind="run", L=12, R=77_777, n_temps=51, beta_max=5.0, n_sweeps=10, n_pop=1,
             eps=0.0, model=0, schedule="optimized", spins=False),
        # a lattice too large for a shared-memory tile
        dict(name="large_lattice", kind="run", L=24, R=20_000, n_temps=11, beta_max=1.0, n_sweeps=10, n_pop=1,
             eps=0.0, model=0, schedule="flat", spins=False),
        # disorder averages: many samples of mixed sizes advanced together
        dict(name="batch_mix", kind="batch", n_runs=64, r_lo=1e4, r_hi=1e5, n_temps=101),
        # requests of mixed sizes handed to a server
        dict(name="served_stream", kind="serve", n_runs=64, r_lo=1e3, r_hi=2e5),
        # the paper's coupling model with both overlaps
        dict(name="gauss_overlap", kind="run", L=8, R=100_000, n_temps=61, beta_max=3.0, n_sweeps=10, n_pop=2,
             eps=0.0, model=1, schedule="flat", spins=False),
        # the paper's coupling model at the paper's schedule
        dict(name="gauss_adaptive", kind="run", L=10, R=1_000_000, n_temps=4096, beta_max=5.0, n_sweeps=10, n_pop=1,
             eps=0.272, model=1, schedule="flat", spins=False),
        # the allocation-free resampling of a caller that owns its device memory
        dict(name="resample_counts", kind="noalloc", n_old=1_000_000, n_levels=3001, spread=0.68),
        # taking a whole population out for analysis
        dict(name="population_read", kind="read", L=10, R=100_000, n_temps=7, n_sweeps=5, model=0),
        # saving a long run and resuming it
        dict(name="checkpoint_resume", kind="checkpoint", L=8, R=50_000, n_temps=9, n_sweeps=5, model=0),
    ]


def _log_uniform(rng: random.Random, lo: float, hi: float) -> int:
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng: random.Random) -> dict:
    kind = rng.choice(["run", "run", "run", "adaptive", "lattice", "gauss", "gauss_adaptive", "batch", "serve",
                       "noalloc", "read", "checkpoint"])
    if kind == "noalloc":
        return dict(kind="noalloc", n_old=_log_uniform(rng, 1, pa.NOALLOC_MAX_SLOTS), spread=rng.uniform(0.0, 2.5),
                    n_levels=3 * rng.choice([4, 6, 8, 10, 12, 16]) ** 3 + 1)
    if kind in ("read", "checkpoint"):
        L = rng.choice([4, 6, 8, 10, 12])
        return dict(kind=kind, L=L, R=_log_uniform(rng, 100, min(1e5, 6e7 / L ** 3)), n_temps=rng.randint(2, 9),
                    n_sweeps=rng.randint(1, 5), model=rng.choice([0, 0, 1]))
    if kind == "batch":
        return dict(kind="batch", n_runs=rng.randint(4, 48), r_lo=1e3, r_hi=float(_log_uniform(rng, 2e3, 1e5)),
                    n_temps=rng.choice([21, 51, 101]))
    if kind == "serve":
        return dict(kind="serve", n_runs=rng.randint(4, 48), r_lo=1e3, r_hi=float(_log_uniform(rng, 2e3, 1e5)))
    adaptive = kind in ("adaptive", "gauss_adaptive")
    gauss = kind in ("gauss", "gauss_adaptive")
    if kind == "lattice":
        L, n_temps, n_sweeps = rng.choice([18, 20, 24, 32]), rng.randint(3, 11), rng.randint(1, 10)
    else:
        L = rng.choice([4, 6, 8, 10, 12] if gauss or adaptive else [2, 4, 6, 8, 10, 12, 14, 16])
        n_temps = 4096 if adaptive else rng.choice([11, 21, 51, 101, 201])
        n_sweeps = rng.randint(5, 10) if adaptive else rng.randint(1, 20)
    n_pop = 1 if adaptive else rng.choice([1, 2])
    beta_max = rng.uniform(0.5, 1.5) if kind == "lattice" else rng.uniform(1.0, 5.0)
    # bounded so that no drawn run costs more than the largest listed ones
    budget = 2e10 if kind == "lattice" else 1e11 if gauss else 2e11
    steps = 90 if adaptive else n_temps
    top = max(200.0, min(1e6, budget / (steps * n_sweeps * n_pop * L ** 3)))
    return dict(kind="run", L=L, R=_log_uniform(rng, 1000 if adaptive else 100, max(top, 2000)), n_temps=n_temps,
                beta_max=beta_max, n_sweeps=n_sweeps, n_pop=n_pop, eps=rng.uniform(0.1, 0.35) if adaptive else 0.0,
                model=1 if gauss else 0, schedule="flat" if adaptive else rng.choice(["flat", "flat", "optimized"]),
                spins=False)


# ---------------------------------------------------------------- inputs

def _seeds(seed: int):
    return (2 * seed + 1) % (1 << 40), (7919 * seed + 1000) % (1 << 40)


def _sweeps(case: dict, betas: np.ndarray) -> Optional[np.ndarray]:
    """Sweeps per step of the optimised schedule: 3 below beta 0.5, 22 up to 2.5, 1 above."""
    if case["schedule"] != "optimized":
        return None
    return np.where(betas < 0.5, 3, np.where(betas <= 2.5, 22, 1)).astype(np.int32)


def _workload(case: dict, seed: int) -> Workload:
    disorder, run = _seeds(seed)
    betas = None if case.get("eps") else linear_betas(case["n_temps"], case.get("beta_max", 1.0))
    return Workload("case", L=case["L"], R=case["R"], disorder_seed=disorder, run_seed=run, betas=betas,
                    n_temps=case["n_temps"], beta_max=case.get("beta_max", 1.0), eps_target=case.get("eps", 0.0),
                    n_sweeps=case["n_sweeps"], n_pop=case.get("n_pop", 1), model=case["model"],
                    sweeps_per_step=_sweeps(case, betas) if "schedule" in case and betas is not None else None)


def _mix(case: dict, seed: int) -> List[Workload]:
    first = (1000 * seed + 100) % (1 << 31)
    if case["kind"] == "batch":
        return batched_mix(case["n_runs"], first_seed=first, n_temps=case["n_temps"], r_lo=case["r_lo"],
                           r_hi=case["r_hi"])
    return [w for w, _ in serving_stream(case["n_runs"], first_seed=first, arrival_seed=seed % (1 << 31),
                                         r_lo=case["r_lo"], r_hi=case["r_hi"])]


def _noalloc_inputs(case: dict, seed: int) -> dict:
    """A population's energy levels, normal about a fifth of the range, and the resampling tables of a
    temperature move dbeta (floor(tau_k) and 2^32 frac(tau_k)); spread is dbeta times the standard
    deviation of the energy: 0.68 culls 27 %, 2.2 is the first step of a coarse linear schedule."""
    rng = np.random.default_rng(seed)
    n, nl = case["n_old"], case["n_levels"]
    sigma = 0.4 * math.sqrt(nl)
    levels = np.clip(np.rint(rng.normal(0.2 * nl, sigma, n)), 0, nl - 1).astype(np.int32)
    w = np.exp(-case["spread"] / sigma * (np.arange(nl) - int(levels.min())))
    w[: int(levels.min())] = 0.0
    tau = n * w / float(np.sum(w[levels]))
    fl = np.floor(tau)
    return dict(levels=levels, fl=fl.astype(np.int32), thr=((tau - fl) * 4294967296.0).astype(np.uint32),
                run_seed=_seeds(seed)[1], t=1 + seed % 50, cap=n + 10 * math.ceil(math.sqrt(n)) + 1024)


def prepare(case: dict, seed: int) -> dict:
    kind = case["kind"]
    state = dict(case=case)
    if kind == "run":
        state["workload"] = _workload(case, seed)
    elif kind == "batch":
        state["workloads"] = _mix(case, seed)
    elif kind == "serve":
        state["workloads"] = _mix(case, seed)
        state["server"] = pa.Server(mem_budget=32 << 30, max_active=256, steps_per_poll=4)
    elif kind == "noalloc":
        inp = _noalloc_inputs(case, seed)
        for k in ("levels", "fl"):
            state[k] = torch.from_numpy(inp[k]).cuda()
        state["thr"] = torch.from_numpy(inp["thr"].view(np.int32)).cuda()
        state["counts"] = torch.zeros(case["n_old"], dtype=torch.int32, device="cuda")
        state["parents"] = torch.full((inp["cap"],), -1, dtype=torch.int32, device="cuda")
        state["n_new"] = torch.zeros(1, dtype=torch.int64, device="cuda")
        state.update(run_seed=inp["run_seed"], t=inp["t"])
    else:  # a run in mid-schedule
        w = _workload(case, seed)
        state["workload"] = w
        state["handle"] = pa.Run.from_workload(w)
        if kind == "read":
            state["handle"].run()
        else:
            for _ in range(case["n_temps"] - 2):
                state["handle"].step()
    return state


# ---------------------------------------------------------------- one pass

# Results come in shapes that do not depend on the seed: per-slot arrays filled up to the population's
# capacity, the rows of an adaptive run to _ROWS.

def _filled(a: np.ndarray, n: int, fill: int) -> np.ndarray:
    out = np.full((n,) + a.shape[1:], fill, dtype=a.dtype)
    out[: len(a)] = a
    return out


def _table(rows: List[dict], n: int = 0) -> dict:
    """Observables as arrays over the rows: the counts in one, every floating-point one by itself."""
    fields = pa.GObs._fields_ if "ql_sum" in rows[0] else pa.Obs._fields_
    floating = [name for name, kind in fields if kind is ctypes.c_double]
    counts = [name for name, kind in fields if kind is not ctypes.c_double]
    out = {"counts": np.array([[r[c] for c in counts] for r in rows], dtype=np.int64)}
    out.update({f: np.array([r[f] for r in rows], dtype=np.float64) for f in floating})
    return {k: _filled(v, max(n, len(rows)), 0) for k, v in out.items()}


def _slots(w: Workload, families, parents, copies, population=None) -> list:
    """The per-slot results of one population: family sizes and their counts, parents, copy numbers and,
    if given, spins, labels and energies."""
    n_sizes = int(math.sqrt(2.0 * w.capacity)) + 2
    return ([_filled(a, n_sizes, 0) for a in families] + [_filled(a, w.capacity, -1) for a in (parents, copies)] +
            [_filled(a, w.capacity, 0) for a in population or []])


def _run(state: dict) -> dict:
    case, w = state["case"], state["workload"]
    gauss = w.model == pa.PA_MODEL_GAUSS
    run = pa.Run.from_workload(w)
    read = run.gobs if gauss else run.obs
    rows: List[List[dict]] = [[] for _ in range(w.n_pop)]
    while True:  # step t's observables are read once step t + 1 has been issued
        t = run.t
        rc = run.step()
        for p in range(w.n_pop):
            rows[p].append(read(t, p))
        if rc == pa.PA_DONE:
            break
    out = {f"obs{p}": _table(rows[p], _ROWS if w.betas is None else 0) for p in range(w.n_pop)}
    t = run.t
    for p in range(w.n_pop):
        out[f"slots{p}"] = _slots(w, run.family_hist(p), run.parents(p), run.copy_counts(p),
                                  run.population(p) if case["spins"] else None)
        out[f"energies{p}"] = _filled(run.genergies(p), w.capacity, 0) if gauss else run.energy_hist(t, p)
    if w.n_pop == 2:
        out["q_hist"] = run.q_hist(t)
        if gauss:
            out["ql_hist"] = run.ql_hist(t)
    run.close()
    return out


def _batch(state: dict) -> dict:
    ws = state["workloads"]
    batch = pa.Batch(ws)
    batch.run()
    views = [batch.run_view(i) for i in range(len(ws))]
    out = {"obs": _table([v.obs(v.t, 0) for v in views]),
           "hist": np.concatenate([v.energy_hist(v.t, 0) for v in views])}
    batch.close()
    return out


def _serve(state: dict) -> dict:
    server = state["server"]
    ids = [server.submit(w) for w in state["workloads"]]
    left = set(ids)
    while left:
        left.difference_update(server.poll())
    results = [server.result(i) for i in ids]
    return {"obs": _table([r[0] for r in results]), "last": np.array([r[1] for r in results])}


def _noalloc(state: dict) -> dict:
    case = state["case"]
    rc = pa.resample_counts_noalloc(state["levels"].data_ptr(), case["n_old"], state["fl"].data_ptr(),
                                    state["thr"].data_ptr(), case["n_levels"], state["run_seed"], 0, state["t"],
                                    state["counts"].data_ptr(), state["parents"].data_ptr(),
                                    state["parents"].numel(), state["n_new"].data_ptr(),
                                    torch.cuda.current_stream())
    if rc != pa.PA_OK:
        raise pa.PAError("pa_resample_counts_noalloc", rc)
    return {"counts": state["counts"], "parents": state["parents"], "n_new": state["n_new"]}


def _checkpoint(state: dict) -> dict:
    saved = state["handle"].checkpoint()
    resumed = pa.Run.from_workload(state["workload"], checkpoint=saved)
    resumed.step()
    w = state["workload"]
    obs = resumed.gobs(resumed.t) if w.model == pa.PA_MODEL_GAUSS else resumed.obs(resumed.t)
    # room for the whole capacity's slots (spins, labels, energies, copies, parents, family sizes) and the records
    room = w.capacity * (w.N + 28) + w.n_temps * (12 * w.N + 2048) + 4096
    out = {"saved": _filled(np.frombuffer(saved, dtype=np.uint8), room, 0), "obs": _table([obs]),
           "slots": _slots(w, resumed.family_hist(), resumed.parents(), resumed.copy_counts())}
    resumed.close()
    return out


def run(state: dict):
    kind = state["case"]["kind"]
    if kind == "run":
        return _run(state)
    if kind == "batch":
        return _batch(state)
    if kind == "serve":
        return _serve(state)
    if kind == "noalloc":
        return _noalloc(state)
    if kind == "read":
        return [_filled(a, state["workload"].capacity, 0) for a in state["handle"].population()]
    return _checkpoint(state)


# ---------------------------------------------------------------- what a pass cannot do without

# Integer operations of one Metropolis update, bit-sliced over 32 replicas: six bond tests, a
# six-input count, a threshold comparison and the flip (about 24 operations), and two random bits
# per replica out of a 40-operation Philox block of 128.
_OPS_PM1 = 24.0 / 32.0 + 2.0 * 40.0 / 128.0
# Gaussian couplings: a threshold per replica (a look-up, a 16-bit uniform, a comparison) beside the bonds.
_OPS_GAUSS = 13.0 / 8.0 + 3.0 + 40.0 / 8.0


def _run_work(w: Workload) -> dict:
    steps = 70 if w.betas is None else len(w.betas) - 1
    sweeps = float(np.sum(w.sweeps_per_step[1:])) if w.sweeps_per_step is not None else float(steps * w.n_sweeps)
    replicas = float(w.R) * w.n_pop
    updates = sweeps * w.N * replicas
    # per step every spin is read and written once (one bit), beside its label, parent and copy number
    per_step = replicas * (2.0 * w.N / 8.0 + 20.0)
    return {"bytes": steps * per_step, "flops": updates * (_OPS_GAUSS if w.model else _OPS_PM1)}


def work(case: dict) -> dict:
    kind = case["kind"]
    if kind == "run":
        return _run_work(_workload(case, 1))
    if kind in ("batch", "serve"):
        parts = [_run_work(w) for w in _mix(case, 1)]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    if kind == "noalloc":
        return {"bytes": 12.0 * case["n_old"], "flops": 20.0 * case["n_old"]}
    N = case["L"] ** 3
    population = case["R"] * (N / 8.0 + 12.0)  # as stored
    written = case["R"] * (N + 12.0)           # as handed over: a byte a spin
    if kind == "read":
        return {"bytes": population + written, "flops": float(case["R"] * N)}
    return {"bytes": 2.0 * (population + written), "flops": case["n_sweeps"] * N * case["R"] * _OPS_PM1}


# ---------------------------------------------------------------- the same in plain numpy and torch

_M32 = 0xFFFFFFFF


def _philox(c0, c1, c2, c3, key):
    """Philox4x32-10 on int64 tensors holding 32-bit words; the counter words broadcast."""
    k0, k1 = key
    for _ in range(10):
        p0, p1 = c0 * 0xD2511F53, c2 * 0xCD9E8D57
        c0, c1, c2, c3 = (((p1 >> 32) & _M32) ^ c1 ^ k0, p1 & _M32, ((p0 >> 32) & _M32) ^ c3 ^ k1, p0 & _M32)
        k0, k1 = (k0 + 0x9E3779B9) & _M32, (k1 + 0xBB67AE85) & _M32
    return c0, c1, c2, c3


def _key(seed: int, purpose: int, pop: int):
    return seed & _M32, (seed >> 32) | (purpose << 28) | (pop << 24)


class _Plain:
    """One population of a +-1 run from the definitions of Amey & Machta: spins [N, R] of 0 / 1 (1 for
    s = -1), with the documented random words."""

    def __init__(self, w: Workload, pop: int):
        self.w, self.dev = w, torch.device("cuda" if torch.cuda.is_available() else "cpu")
        self.pop, L, N = pop, w.L, w.N
        n = self.words(torch.arange(N))
        j = _philox(n, n * 0, n * 0, n * 0, _key(w.disorder_seed, 0, 0))
        self.J = torch.stack([v & 1 for v in j[:3]], 1)  # 1 for J = -1
        x, y, z = n % L, n // L % L, n // (L * L)
        site = lambda a, b, c: a % L + L * (b % L + L * (c % L))
        self.fwd = torch.stack([site(x + 1, y, z), site(x, y + 1, z), site(x, y, z + 1)], 1)
        self.bwd = torch.stack([site(x - 1, y, z), site(x, y - 1, z), site(x, y, z - 1)], 1)
        self.colour = [torch.nonzero((x + y + z) % 2 == c).flatten() for c in (0, 1)]
        r = self.words(torch.arange((w.R + 3) // 4))
        init = _philox(n[:, None], n[:, None] * 0, r[None, :], r[None, :] * 0, _key(w.run_seed, 1, pop))
        self.s = torch.stack([v & 1 for v in init], 2).reshape(N, -1)[:, : w.R].contiguous()
        self.labels = torch.arange(w.R, device=self.dev)
        self.betas, self.lnq, self.E0, self.rows = [0.0], [], 1 << 30, []
        self.parents = self.copies = None
        self.measure(0, 0.0, {})

    def words(self, a):
        return a.to(self.dev, torch.int64)

    def levels(self):
        k = torch.zeros(self.s.shape[1], dtype=torch.int64, device=self.dev)
        for d in range(3):
            k += (self.s ^ self.s[self.fwd[:, d]] ^ self.J[:, d, None]).sum(0)
        return k

    def measure(self, t: int, dbeta: float, resampled: dict):
        w, R = self.w, self.s.shape[1]
        self.k = self.levels()
        self.hist = torch.bincount(self.k, minlength=3 * w.N + 1).cpu().numpy()
        E = 2 * np.arange(3 * w.N + 1, dtype=np.int64) - 3 * w.N
        sE, sE2, Emin = int((self.hist * E).sum()), int((self.hist * E * E).sum()), int(E[self.hist > 0].min())
        self.E0 = min(self.E0, Emin)
        self.eta = torch.unique_consecutive(self.labels, return_counts=True)[1].cpu().numpy()
        nu = self.eta / R
        S_f = -math.fsum(nu * np.log(nu))
        mbF = w.N * math.log(2.0) + math.fsum(self.lnq)
        s2 = int((self.eta.astype(np.int64) ** 2).sum())
        row = dict(t=t, beta=self.betas[-1], dbeta=dbeta, R_tilde=R, sum_E=sE, sum_E2=sE2, E_min=Emin,
                   mean_E=sE / R, var_E=sE2 / R - (sE / R) ** 2, kmin_prev=0, S_prime=0.0, lnQ=0.0, minus_beta_F=mbF,
                   eps_expected=0.0, culled=0, sum_eta2=s2, n_families=len(self.eta), rho_t=s2 / R, S_f=S_f,
                   rho_s=R / math.exp(S_f), E0=self.E0, g0_tilde=int(self.hist[(self.E0 + 3 * w.N) // 2]) / R,
                   g0_bar=2.0 * math.exp(-(self.betas[-1] * self.E0) - mbF), q_pairs=0, q_abs_le_02=0, I02=0.0)
        row.update(resampled)
        self.rows.append(row)

    def weights(self, dbeta: float):
        occ = np.nonzero(self.hist)[0]
        w = [math.exp(-(dbeta * float(2 * (k - occ[0])))) for k in occ]
        S = 0.0
        for k, v in zip(occ, w):
            S = S + float(self.hist[k]) * v
        return occ, w, S

    def culling(self, dbeta: float) -> float:
        occ, w, S = self.weights(dbeta)
        eps = 0.0
        for k, v in zip(occ, w):
            tau = (float(self.w.R) * v) / S
            if tau < 1.0:
                eps = eps + float(self.hist[k]) * (1.0 - tau)
        return eps / float(self.w.R)

    def choose(self) -> float:
        """The largest move whose culling fraction stays within the target, by 64 halvings."""
        rem = self.w.beta_max - self.betas[-1]
        if self.culling(rem) <= self.w.eps_target:
            return rem
        lo, hi = 0.0, rem
        for _ in range(64):
            mid = 0.5 * (lo + hi)
            lo, hi = (mid, hi) if self.culling(mid) <= self.w.eps_target else (lo, mid)
        return lo if lo > 0.0 else hi

    def step(self, t: int, beta: float, n_sweeps: int):
        w, R = self.w, self.s.shape[1]
        dbeta = beta - self.betas[-1]
        occ, wt, S = self.weights(dbeta)
        fl, thr = np.zeros(3 * w.N + 1, dtype=np.int64), np.zeros(3 * w.N + 1, dtype=np.int64)
        for k, v in zip(occ, wt):
            tau = (float(w.R) * v) / S
            fl[k], thr[k] = int(math.floor(tau)), int((tau - math.floor(tau)) * 4294967296.0)
        g = self.words(torch.arange((R + 3) // 4))
        r = torch.stack(_philox(g, g * 0, g * 0, g * 0 + t, _key(w.run_seed, 3, self.pop)), 1).flatten()[:R]
        self.copies = self.words(torch.from_numpy(fl))[self.k] + (r < self.words(torch.from_numpy(thr))[self.k])
        self.parents = torch.repeat_interleave(torch.arange(R, device=self.dev), self.copies)
        kmin, E_low = int(occ[0]), 2 * int(occ[0]) - 3 * w.N
        lnq = math.log(S / R) - dbeta * E_low
        done = dict(kmin_prev=kmin, S_prime=S, lnQ=lnq, eps_expected=self.culling(dbeta),
                    culled=int((self.copies == 0).sum()))
        self.lnq.append(lnq)
        self.s, self.labels = self.s[:, self.parents], self.labels[self.parents]
        self.betas.append(beta)
        self.sweep(t, beta, n_sweeps)
        self.measure(t, dbeta, done)

    def sweep(self, t: int, beta: float, n_sweeps: int):
        R = self.s.shape[1]
        acc = [min(int(math.floor(math.ldexp(math.exp(-(beta * 4.0 * m)), 32))), _M32) for m in (3, 2, 1)]
        thr = torch.tensor(acc + [1 << 32] * 4, device=self.dev)  # by unsatisfied bonds; three or more always flip
        groups = self.words(torch.arange((R + 31) // 32))
        bit = torch.arange(32, device=self.dev)
        for s in range(n_sweeps):
            for c in (0, 1):
                n = self.colour[c]
                u = torch.zeros(len(n), R, dtype=torch.int64, device=self.dev)
                for d in range(3):
                    u += self.s[n] ^ self.s[self.fwd[n, d]] ^ self.J[n, d, None]
                    u += self.s[n] ^ self.s[self.bwd[n, d]] ^ self.J[self.bwd[n, d], d, None]
                # plane p of the uniforms: bit 31 - p of replica j is bit j mod 32 of its group's word
                h, U = (n >> 1)[:, None, None], 0
                block = 8 * groups[None, :, None] + self.words(torch.arange(8))[None, None, :]
                w4 = _philox(h, h * 0 + 2 * s + c, block, h * 0 + t, _key(self.w.run_seed, 2, self.pop))
                for p in range(32):
                    U = U + (((w4[p % 4][:, :, p // 4, None] >> bit) & 1) << (31 - p))
                self.s[n] ^= (U.reshape(len(n), -1)[:, :R] < thr[u]).to(torch.int64)


def _exact_run(case: dict, seed: int):
    w = _workload(case, seed)
    steps = 90 if w.betas is None else len(w.betas) - 1
    sweeps = float(np.sum(w.sweeps_per_step)) if w.sweeps_per_step is not None else float(steps * w.n_sweeps)
    if w.model or 2.0 * w.n_pop * sweeps * (0.008 + 130.0 * 24.0 * w.N / 2 * w.R / 4e12) > 18.0:
        return None
    pops = [_Plain(w, p) for p in range(w.n_pop)]
    q_rows = []
    for t in range(w.n_temps):
        if t > 0:
            beta = pops[0].betas[-1] + pops[0].choose() if w.betas is None else float(w.betas[t])
            if w.betas is None and beta >= w.beta_max:
                beta = w.beta_max
            S_t = int(w.sweeps_per_step[t]) if w.sweeps_per_step is not None else w.n_sweeps
            for p in pops:
                p.step(t, beta, S_t)
        if w.n_pop == 2:
            R = min(p.s.shape[1] for p in pops)
            Q = (w.N - 2 * (pops[0].s[:, :R] ^ pops[1].s[:, :R]).sum(0)).cpu().numpy()
            q_rows.append(np.bincount(((Q + w.N) * (w.q_bins - 1) + w.N) // (2 * w.N), minlength=w.q_bins))
            low = int((5 * np.abs(Q) <= w.N).sum())
            for p in pops:
                p.rows[-1].update(q_pairs=R, q_abs_le_02=low, I02=low / R)
        if w.betas is None and pops[0].betas[-1] >= w.beta_max:
            break
    out = {f"obs{i}": _table(p.rows, _ROWS if w.betas is None else 0) for i, p in enumerate(pops)}
    for i, p in enumerate(pops):
        families = [a.astype(np.int64) for a in np.unique(p.eta, return_counts=True)]
        population = [(1 - 2 * p.s.T).cpu().numpy().astype(np.int8), p.labels.cpu().numpy().astype(np.int32),
                      (2 * p.k - 3 * w.N).cpu().numpy().astype(np.int32)]
        out[f"slots{i}"] = _slots(w, families, p.parents.cpu().numpy().astype(np.int32),
                                  p.copies.cpu().numpy().astype(np.int32), population if case["spins"] else None)
        out[f"energies{i}"] = p.hist.astype(np.int64)
    if w.n_pop == 2:
        out["q_hist"] = q_rows[-1].astype(np.int64)
    return out


def _exact_noalloc(case: dict, seed: int):
    inp = _noalloc_inputs(case, seed)
    n = case["n_old"]
    g = torch.arange((n + 3) // 4)
    r = torch.stack(_philox(g, g * 0, g * 0, g * 0 + inp["t"], _key(inp["run_seed"], 3, 0)), 1).flatten()[:n].numpy()
    counts = inp["fl"][inp["levels"]] + (r < inp["thr"].astype(np.int64)[inp["levels"]])
    parents = np.full(inp["cap"], -1, dtype=np.int32)
    made = np.repeat(np.arange(n, dtype=np.int32), counts)[: inp["cap"]]
    parents[: len(made)] = made
    return {"counts": counts.astype(np.int32), "parents": parents,
            "n_new": np.array([counts.sum()], dtype=np.int64)}


def exact(case: dict, seed: int):
    if case["kind"] == "run":
        return _exact_run(case, seed)
    if case["kind"] == "noalloc":
        return _exact_noalloc(case, seed)
    return None
