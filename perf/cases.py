"""The framework's work as its users have it done: which calls, on which sizes.

A case is a dict of plain values; prepare() makes the engine (or the server, or
the host records) that a program keeps, run() is one pass through the public
entry points and returns what the pass computes, work() counts what the pass
cannot do without, and exact() gives the floating-point results of the smaller
cases from a plain torch / numpy restatement of the method in 64 bits.

Three kinds of case:
  anneal  a batch of runs through some or all temperatures of their schedules,
          then the records, the weighted averages or the population read back
  serve   jobs through a server engine with fewer slots than jobs
  wavg    free-energy-weighted averages of records held on the host
"""
import functools
import math

import numpy as np
import torch

from paper_2207_05535_gb300 import _lib, dos, serve
from paper_2207_05535_gb300 import workloads as W

# Per attempted spin update: a quarter of a Philox4x32-10 call (20 multiplies and 20
# three-input xors) and the acceptance test.
OPS_PER_UPDATE = 11
REC_BYTES = _lib.RECORD_DTYPE.itemsize
WAVG_BYTES = _lib.WAVG_DTYPE.itemsize

ANNEAL = dict(kind="anneal", model="fm", theta=10, beta_f=1.0, resample="nearest", overlap="none", group=0,
              read="records", population="none")


def listed():
    return [
        # One interactive run: a single small ferromagnet from start to finish, its records
        # and its configurations; nothing but latency.
        dict(ANNEAL, name="single_L16", L="16", R="1000", runs=1, beta_f=0.5, temps=21, steps=20, population="all"),
        # The small benchmark batch: 20 ferromagnet runs, their whole anneal and weighted averages.
        dict(ANNEAL, name="ising_L8_batch", L="8", R="500", runs=20, beta_f=0.5, temps=51, steps=50, group=20),
        # Weighted averages at their purpose: very many populations far too small by themselves.
        dict(ANNEAL, name="many_small_L16", L="16", R="100", runs=2048, theta=2, beta_f=0.5, temps=51, steps=50,
             group=64, read="last"),
        # The glass benchmark: 100 disorder samples of two populations, both overlaps, whole anneal.
        dict(ANNEAL, name="glass_L16_pairs", model="ea", L="16", R="5000", runs=200, beta_f=3.0, temps=101,
             steps=100, overlap="shift+pair", group=2),
        # An uneven batch of lattice and population sizes in one engine, part of its schedule.
        dict(ANNEAL, name="uneven_batch", L="16,32,64,128", R="1000,10000,50000", runs=48, temps=101, steps=8,
             read="last", population="energies"),
        # One large lattice with a large population, part of its schedule.
        dict(ANNEAL, name="ising_L256", L="256", R="100000", runs=1, theta=20, beta_f=0.44, temps=201, steps=8,
             population="energies"),
        # Lattice sizes that are not powers of two, ferromagnets and glasses side by side.
        dict(ANNEAL, name="ragged_mixed", model="mixed", L="30,46,100", R="10000,3333", runs=24, temps=41, steps=12,
             population="energies"),
        # A server with fewer slots than jobs: even L from 8 to 64, both models, continuous batching.
        dict(kind="serve", name="server_mixed", jobs=32, slots=16, Lmin=8, Lmax=64, Rmin=1000, Rmax=50000, nmin=12,
             nmax=40, theta=10, mix=11),
        # theta = infinity: energies drawn from the exact density of states, whole anneal.
        dict(ANNEAL, name="theta_inf_L8", model="dos", L="8", R="20000", runs=200, theta=0, beta_f=0.6, temps=61,
             steps=60),
        # Multinomial resampling (constant population size).
        dict(ANNEAL, name="multinomial_L16", L="16", R="10000", runs=20, beta_f=0.5, temps=31, steps=30,
             resample="multinomial"),
        # Glass overlaps over random pairings that keep families apart.
        dict(ANNEAL, name="wang_L16", model="ea", L="16", R="4000", runs=20, beta_f=1.5, temps=16, steps=15,
             overlap="wang"),
        # Records of earlier runs combined on the device, with the overlap distribution.
        dict(kind="wavg", name="wavg_host", M=200, temps=101, L=16, R=5000, qhist=True, weight=0),
    ]


def draw(rng):
    """One more case of the same kinds; at most about 3e11 attempted updates (the largest listed one: 1e12)."""
    kind = rng.choice(["fm", "fm", "ea", "ragged", "mixed", "dos", "multinomial", "wang", "serve", "wavg"])

    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    if kind == "serve":
        jobs = rng.randint(4, 40)
        return dict(kind="serve", jobs=jobs, slots=rng.randint(2, jobs), Lmin=8, Lmax=2 * rng.randint(8, 32),
                    Rmin=1000, Rmax=log_int(2000, 30000), nmin=11, nmax=rng.randint(16, 40), theta=10,
                    mix=rng.randint(0, 10**6))
    if kind == "wavg":
        M, L = log_int(2, 500), 2 * rng.randint(4, 12)
        temps = rng.randint(11, 101)
        return dict(kind="wavg", M=M, temps=temps, L=L, R=log_int(100, 50000), weight=rng.randint(0, 1),
                    qhist=bool(rng.randint(0, 1)) and M * temps * L * L < 10**7)
    steps = rng.randint(10, 40)
    c = dict(ANNEAL, temps=steps + 1, steps=steps, theta=rng.choice([1, 2, 5, 10, 20]),
             beta_f=round(rng.uniform(0.02, 0.05) * steps, 3))
    R = log_int(60, 40000)
    if kind == "dos":
        c.update(model="dos", L=str(rng.choice([4, 6, 8])), theta=0, beta_f=0.6)
        runs = max(1, min(300, log_int(10**5, 10**8) // (R * steps)))
    else:
        if kind == "fm" or kind == "multinomial":
            L = rng.choice([8, 16, 32, 64, 128, 256] if kind == "fm" else [8, 16, 22, 32])
            c.update(model="fm")
        elif kind == "ea" or kind == "wang":
            L = rng.choice([8, 16, 32, 64] if kind == "ea" else [8, 12, 16, 20])
            c.update(model="ea", overlap="wang" if kind == "wang" else rng.choice(["none", "shift+pair"]))
        else:
            L = rng.choice([4, 6, 10, 12, 14, 18, 20, 22, 24, 26, 30, 34, 38, 40, 46, 48, 54, 60, 66, 80, 100, 120])
            c.update(model=rng.choice(["fm", "ea"]) if kind == "ragged" else "mixed")
        c.update(L=str(L))
        if kind == "multinomial":
            c.update(resample="multinomial")
        if kind == "wang":
            R = min(R, 7000)
        runs = max(1, min(400, log_int(10**7, 3 * 10**11) // (R * L * L * c["theta"] * steps)))
        if R * L * L * c["theta"] * steps > 3 * 10**11:
            R = max(50, int(3e11 / (L * L * c["theta"] * steps)))
    if c["overlap"] == "shift+pair":
        runs = 2 * ((runs + 1) // 2)
    c.update(R=str(R), runs=runs, read=rng.choice(["records", "last"]))
    if kind in ("fm", "multinomial") and runs > 1:
        c.update(group=rng.choice([0, runs]))
    if runs == 1 and R * int(c["L"]) ** 2 < 10**7 and c["model"] != "dos":
        c.update(population="all")
    elif rng.randint(0, 1):
        c.update(population="energies")
    return c


@functools.lru_cache(maxsize=None)
def _log_g(L):
    return dos.log_dos(L)


def _ints(text):
    return [int(x) for x in text.split(",")]


def _descs(case, seed):
    """The run descriptors of an anneal case: sizes from the case alone, randomness keyed by the seed."""
    Ls, Rs = _ints(case["L"]), _ints(case["R"])
    betas = W.schedule(case["beta_f"], case["temps"])
    overlap = {"none": W.Q_NONE, "shift+pair": W.Q_SHIFT | W.Q_PAIR, "wang": W.Q_WANG}[case["overlap"]]
    key = seed % (1 << 32)
    out = []
    for k in range(case["runs"]):
        L, R = Ls[k % len(Ls)], Rs[(k // len(Ls)) % len(Rs)]
        model = {"fm": 0, "dos": 0, "ea": 1, "mixed": k // len(Ls) % 2}[case["model"]]
        pair = bool(overlap & W.Q_PAIR)
        out.append(W.RunDesc(L, W.EA_PMJ if model else W.FERRO, R,
                             W.THETA_INF if case["model"] == "dos" else case["theta"], betas, key, k,
                             k // 2 if pair else k, W.MULTINOMIAL if case["resample"] == "multinomial" else W.NEAREST,
                             overlap, k ^ 1 if pair else -1, log_g=_log_g(L) if case["model"] == "dos" else None))
    return out


def _jobs(case, seed):
    rng = np.random.default_rng(case["mix"])
    out = []
    for m in range(case["jobs"]):
        model = int(rng.integers(0, 2))
        L = int(2 * rng.integers(case["Lmin"] // 2, case["Lmax"] // 2 + 1))
        R = int(round(math.exp(rng.uniform(math.log(case["Rmin"]), math.log(case["Rmax"])))))
        n = int(rng.integers(case["nmin"], case["nmax"] + 1))
        # the jobs anneal with the step of a full-length schedule
        out.append(W.RunDesc(L, model, R, case["theta"], W.schedule((1.0 if model == W.FERRO else 3.0) * n / 100, n),
                             seed % (1 << 32), m, m))
    return out


def _host_records(case, seed):
    """Records of M runs as earlier anneals left them: energies that fall with beta,
    populations that fluctuate about R, free energies that differ between runs."""
    rng = np.random.default_rng(seed)
    M, n, N, R = case["M"], case["temps"], case["L"] ** 2, case["R"]
    beta = W.schedule(3.0, n)
    rec = np.zeros((M, n), dtype=_lib.RECORD_DTYPE)
    Ri = np.maximum(1, R + np.rint(rng.normal(0, 0.5 * math.sqrt(R), (M, n)))).astype(np.int64)
    Ri[:, 0] = R
    e = -1.4 * np.tanh(1.2 * beta)[None] + rng.normal(0, 0.004, (M, n))
    m = 0.05 + 0.02 * np.tanh(beta)[None] + np.abs(rng.normal(0, 0.002, (M, n)))
    ve, vm = 2.0 / N / (1 + beta[None] ** 2), np.full((M, n), 0.3 / N)
    rec["beta"] = beta[None]
    lnQ = -np.diff(beta, prepend=0.0)[None] * N * e + rng.normal(0, 0.05, (M, n))
    lnQ[:, 0] = 0.0
    rec["lnQ"] = lnQ
    rec["minus_betaF"] = N * math.log(2.0) + np.cumsum(lnQ, axis=1)

    def total(x, power):  # integer sums over the population
        return np.rint(x * float(N) ** power * Ri).astype(np.int64)

    def wide(x):
        return np.stack([x.astype(np.uint64), np.where(x < 0, -1, 0).astype(np.int64).astype(np.uint64)], axis=-1)

    rec["sumE"], rec["sumE2"] = total(e, 1), total(e * e + ve, 2)
    rec["sumAbsM"], rec["sumM2"] = total(m, 1), total(m * m + vm, 2)
    rec["sumE3"], rec["sumE4"] = wide(total(e**3 + 3 * e * ve, 3)), wide(total(e**4 + 6 * e * e * ve + 3 * ve**2, 4))
    rec["sumAbsM3"], rec["sumM4"] = wide(total(m**3 + 3 * m * vm, 3)), wide(total(m**4 + 6 * m * m * vm + 3 * vm**2, 4))
    rec["sum_c2"], rec["n_fam"], rec["max_fam"] = Ri * 3, np.maximum(1, Ri // 2), 7
    rec["R"], rec["R_target"], rec["N"], rec["n_q"] = Ri, R, N, Ri // 2
    rec["sum_absq"] = np.rint(0.3 * N * (Ri // 2)).astype(np.int64)
    qh = None
    if case["qhist"]:
        d = np.arange(N + 1)
        p = np.exp(-0.5 * ((d - 0.35 * N) / (0.08 * N)) ** 2) + np.exp(-0.5 * ((d - 0.65 * N) / (0.08 * N)) ** 2)
        qh = rng.poisson(p / p.sum() * (R // 2), (M, n, N + 1)).astype(np.uint32)
    return rec, qh


class _Anneal:
    """An engine, its case, and its release with the state that holds it."""

    def __init__(self, case, seed):
        self.case = case
        self.eng = _lib.Engine(_descs(case, seed))
        self.ids = np.arange(case["runs"], dtype=np.uint32)


class _Serve:
    def __init__(self, case, seed):
        self.case = case
        self.jobs = _jobs(case, seed)
        self.server = serve.Server(serve.config_for_budget(6 << 30, max_runs=case["slots"], min_L=case["Lmin"],
                                                           max_L=case["Lmax"], max_n_beta=case["nmax"],
                                                           table_bytes=64 << 20))

    def __del__(self):
        if getattr(self, "server", None):
            self.server.close()


def prepare(case, seed):
    if case["kind"] == "anneal":
        return _Anneal(case, seed)
    if case["kind"] == "serve":
        return _Serve(case, seed)
    return case, _host_records(case, seed)


def _split(rec):
    """Records as two plain arrays: (beta, ln Q, -beta F) and the integer words."""
    flat = np.ascontiguousarray(rec)
    words = REC_BYTES // 8
    return {"floats": flat.view("f8").reshape(rec.shape + (words,))[..., :3],
            "whole": flat.view("i8").reshape(rec.shape + (words,))[..., 3:]}


def _floats(w):
    return np.ascontiguousarray(w).view("f8").reshape(w.shape + (WAVG_BYTES // 8,))


def _populations(eng, spins):
    """Every run's replicas as they stand, one run after another, each padded to its capacity with zeros."""
    cap = [r.R_cap for r in eng.runs]
    E, M, fam = (np.zeros(sum(cap), t) for t in (np.int32, np.int32, np.uint32))
    out, at = {"E": E, "M": M, "family": fam}, 0
    for k, r in enumerate(eng.runs):
        if spins:
            s, e, m, f, _ = eng.population(k)
            out["spins"] = np.zeros((cap[k], r.N), np.int8)  # one run
            out["spins"][:len(s)] = s
        else:
            _, e, m, f, _, _ = _lib.pa_population_slice(eng.h, k, 0, cap[k], r.N, spins=False)
        E[at:at + len(e)], M[at:at + len(e)], fam[at:at + len(e)] = e, m, f
        at += cap[k]
    return out


def run(state):
    if isinstance(state, _Anneal):
        case, eng = state.case, state.eng
        eng.reset()
        eng.step(case["steps"])
        eng.sync()
        if case["read"] == "records":
            out = _split(np.stack([eng.records(k)[:case["steps"] + 1] for k in range(case["runs"])]))
        else:
            out = _split(eng.step_records(state.ids))
        if case["group"]:
            w = eng.weighted_average(state.ids, case["group"], W_FULL, q="shift" in case["overlap"])
            out["wavg"] = _floats(w[0] if isinstance(w, tuple) else w)
            if isinstance(w, tuple):
                out["Pq"], out["Pq_pair"] = w[1], w[2]
        if case["population"] != "none":
            out.update(_populations(eng, case["population"] == "all"))
        return out
    if isinstance(state, _Serve):
        queue = [serve.Job(d, 0.0) for d in state.jobs]
        waiting, done = list(queue), 0
        while done < len(queue):
            while waiting and state.server.try_admit(waiting[0]):
                waiting.pop(0)
            state.server.step()
            done += len(state.server.collect())
        return _split(np.concatenate([j.records for j in queue]))
    case, (rec, qh) = state
    out, Pq, _ = _lib.pa_weighted_average(rec, case["L"] ** 2, case["weight"], qh)
    return {"wavg": _floats(out)} if Pq is None else {"wavg": _floats(out), "Pq": Pq}


W_FULL = 0  # weights of Eq. appropriateWeight


def work(case):
    if case["kind"] == "wavg":
        n = case["M"] * case["temps"]
        N = case["L"] ** 2
        q = case["temps"] * (N + 1) if case["qhist"] else 0
        return {"bytes": n * REC_BYTES + case["temps"] * WAVG_BYTES + 4 * case["M"] * q + 8 * q,
                "flops": 60 * n + 2 * case["M"] * q}
    runs = _jobs(case, 0) if case["kind"] == "serve" else None
    if runs is None:
        Ls, Rs = _ints(case["L"]), _ints(case["R"])
        sizes = [(Ls[k % len(Ls)], Rs[(k // len(Ls)) % len(Rs)], case["steps"], case["theta"])
                 for k in range(case["runs"])]
    else:
        sizes = [(d.L, d.R, d.n_beta - 1, d.theta) for d in runs]
    nbytes = ops = 0
    for L, R, steps, theta in sizes:
        N = L * L
        dosrun = case.get("model") == "dos"
        # the beta_0 population and the last one (bit spins, E, M, family), and the records
        nbytes += 2 * R * ((0 if dosrun else N // 8) + 12) + REC_BYTES * (steps + 1)
        # theta = infinity: one Philox call and a search per draw; else theta sweeps; one call per copy number
        ops += R * steps * (40 + (60 if dosrun else theta * N * OPS_PER_UPDATE))
        if case.get("overlap", "none") != "none":
            nbytes += 8 * (steps + 1) * (N + 1)
            ops += R * steps * (N // 16)
    return {"bytes": nbytes, "flops": ops}


# ---- the method restated in 64 bits --------------------------------------

MASK = 0xFFFFFFFF


def _philox(c0, c1, c2, c3, k0, k1):
    """Philox4x32-10 on int64 tensors or ints holding 32-bit values."""
    for r in range(10):
        if r:
            k0, k1 = (k0 + 0x9E3779B9) & MASK, (k1 + 0xBB67AE85) & MASK
        p0, p1 = 0xD2511F53 * c0, 0xCD9E8D57 * c2
        c0, c1, c2, c3 = ((p1 >> 32) & MASK) ^ c1 ^ k0, p1 & MASK, ((p0 >> 32) & MASK) ^ c3 ^ k1, p0 & MASK
    return c0, c1, c2, c3


class _Population:
    """All replicas of a batch of runs of one lattice size, as flat tensors."""

    def __init__(self, descs, dev):
        d = descs[0]
        self.descs, self.dev, self.L, self.N = descs, dev, d.L, d.N
        self.R0 = torch.tensor([x.R for x in descs], device=dev)
        self.seed = d.seed
        self.run = torch.repeat_interleave(torch.arange(len(descs), device=dev), self.R0)
        self.ids = torch.tensor([x.run_id for x in descs], device=dev)
        self.betas = d.betas
        self.theta_inf = d.theta == W.THETA_INF
        L, N = self.L, self.N
        n = torch.arange(N, device=dev)
        self.colour = ((n % L + n // L) & 1).reshape(L, L)
        self.key = self.ids[self.run]
        if self.theta_inf:
            self.E = self._dos(0)
            self.M = torch.zeros_like(self.E)
            return
        u = self._words((n // 4)[None, ::4], self._index()[:, None], 0, 1 << 24)
        self.s = ((u >> 31) * 2 - 1).reshape(-1, L, L).to(torch.int8)
        dis = torch.tensor([x.disorder_id for x in descs], device=dev)[:, None]
        w = torch.stack(torch.broadcast_tensors(*_philox((n // 4)[None, ::4] + 0 * dis, 0 * dis, 0 * dis, (5 << 24) + 0 * dis,
                                                         self.seed, dis)), -1).reshape(-1, N)
        glass = torch.tensor([x.model == W.EA_PMJ for x in descs], device=dev)[:, None]
        one = torch.ones_like(w)
        self.Jr = torch.where(glass, ((w >> 31) & 1) * 2 - 1, one).reshape(-1, L, L).to(torch.int8)
        self.Jd = torch.where(glass, ((w >> 30) & 1) * 2 - 1, one).reshape(-1, L, L).to(torch.int8)
        self._energies()

    def _index(self):
        """Replica index within its run."""
        count = torch.bincount(self.run, minlength=len(self.descs))
        first = torch.cumsum(count, 0) - count
        return torch.arange(len(self.run), device=self.dev) - first[self.run]

    def _words(self, c0, c1, c2, c3):
        w = _philox(c0 + 0 * c1, c1 + 0 * c0, c2 + 0 * c1, c3 + 0 * c1, self.seed, self.key[:, None])
        return torch.stack(torch.broadcast_tensors(*w), -1).flatten(1)

    def _field(self, Jr, Jd):
        s = self.s
        return (Jr * torch.roll(s, -1, 2) + torch.roll(Jr * s, 1, 2) + Jd * torch.roll(s, -1, 1) +
                torch.roll(Jd * s, 1, 1))

    def _energies(self):
        h = self._field(self.Jr[self.run], self.Jd[self.run])
        self.E = -((self.s * h).sum((1, 2), dtype=torch.int64) // 2)
        self.M = self.s.sum((1, 2), dtype=torch.int64)

    def _unit53(self, w0, w1):
        return (((w0 >> 5) << 26) | (w1 >> 6)).double() * 2.0**-53

    def _dos(self, i):
        d = self.descs[0]
        g = torch.tensor(d.log_g, dtype=torch.float64)
        l = g - float(self.betas[i]) * (2.0 * torch.arange(2 * self.N + 1, dtype=torch.float64) - 2.0 * self.N)
        C = torch.cumsum(torch.exp(l - l.max()), 0)
        last = int(torch.nonzero(torch.exp(l - l.max()) > 0).max())
        j = self._index()
        w = _philox(j, 0 * j, i + 0 * j, (6 << 24) + 0 * j, self.seed, self.key)
        lev = torch.searchsorted(C.to(self.dev), self._unit53(w[0], w[1]) * float(C[-1]), right=True)
        return 2 * torch.clamp(lev, max=last) - 2 * self.N

    def resample(self, i):
        """ln Q of every run, and the population replaced by its copies."""
        nr, N, dev = len(self.descs), self.N, self.dev
        db = float(self.betas[i]) - float(self.betas[i - 1])
        low = torch.full((nr,), 1 << 40, device=dev).scatter_reduce(0, self.run, self.E, "amin")
        n = (self.E - low[self.run]) // 4
        w = torch.exp(-db * 4.0 * torch.arange(N + 1, device=dev, dtype=torch.float64))
        h = torch.bincount(self.run * (N + 1) + n, minlength=nr * (N + 1)).reshape(nr, N + 1)
        C = torch.cumsum(h.double() * w, 1)
        S, count = C[:, -1], h.sum(1)
        lnQ = -db * low.double() + torch.log(S) - torch.log(count.double())
        j = self._index()
        if self.descs[0].resample == W.NEAREST:
            tau = self.R0[self.run].double() * w[n] / S[self.run]
            u = _philox(j, 0 * j, i + 0 * j, (3 << 24) + 0 * j, self.seed, self.key)[0]
            r = torch.floor(tau).long() + (u.double() * 2.0**-32 < tau - torch.floor(tau)).long()
        else:
            R = int(self.R0[0])
            k = torch.arange(R, device=dev)[None] + 0 * self.ids[:, None]
            u = _philox(k, 0 * k, i + 0 * k, (4 << 24) + 0 * k, self.seed, self.ids[:, None])
            lev = torch.searchsorted(C, self._unit53(u[0], u[1]) * S[:, None], right=True)
            top = (N - torch.argmax((h.flip(1) > 0).long(), 1))[:, None]
            lev = torch.minimum(lev, top)
            pick = (u[2] * torch.gather(h, 1, lev)) >> 32
            begin = (torch.cumsum(h.flatten(), 0) - h.flatten()).reshape(nr, N + 1)
            members = torch.argsort(self.run * (N + 1) + n, stable=True)
            r = torch.bincount(members[(torch.gather(begin, 1, lev) + pick).flatten()], minlength=len(self.run))
        parent = torch.repeat_interleave(torch.arange(len(r), device=dev), r)
        self.run, self.key = self.run[parent], self.key[parent]
        if not self.theta_inf:
            self.s = self.s[parent]
        return lnQ

    def equilibrate(self, i):
        if self.theta_inf:
            self.E = self._dos(i)
            self.M = torch.zeros_like(self.E)
            return
        beta, L, N, dev = float(self.betas[i]), self.L, self.N, self.dev
        T = [min(1 << 32, int(math.exp(-4.0 * m * beta) * 2.0**32)) for m in (1, 2)]
        T = torch.tensor([1 << 32] * 3 + T, device=dev)  # by dE / 4 + 2
        Jr, Jd = self.Jr[self.run], self.Jd[self.run]
        j = self._index()[:, None]
        k = torch.arange((N // 2 + 3) // 4, device=dev)[None]
        site = (torch.arange(N, device=dev) // 2).reshape(L, L)  # y L/2 + (x >> 1)
        for t in range(self.descs[0].theta):
            for c in range(2):
                u = self._words(k, j, i, (2 << 24) | (t << 1) | c)[:, site.flatten()].reshape(-1, L, L)
                dE = (2 * self.s * self._field(Jr, Jd)).long()
                flip = (u < T[dE // 4 + 2]) & (self.colour == c)
                self.s = torch.where(flip, -self.s, self.s)
        self._energies()

    def sums(self):
        """Per run: R_i and the sums of E, E^2, E^3, E^4, |M|, M^2, |M|^3, M^4 (exact in int64 for L <= 32)."""
        nr = len(self.descs)
        out = [torch.bincount(self.run, minlength=nr)]
        for x in (self.E, self.M.abs()):
            for p in (1, 2, 3, 4):
                out.append(torch.zeros(nr, dtype=torch.int64, device=self.dev).index_add_(0, self.run, x**p))
        return torch.stack(out, 1).double().cpu().numpy()


def _simulate(descs, steps):
    """(beta, ln Q, -beta F) [runs][steps + 1][3] and the sums [runs][steps + 1][9]."""
    pop = _Population(descs, torch.device("cuda" if torch.cuda.is_available() else "cpu"))
    lnQ, sums = [np.zeros(len(descs))], [pop.sums()]
    for i in range(1, steps + 1):
        lnQ.append(pop.resample(i).cpu().numpy())
        pop.equilibrate(i)
        sums.append(pop.sums())
    lnQ = np.stack(lnQ, 1)
    mbF = descs[0].N * math.log(2.0) + np.cumsum(lnQ, 1)
    beta = np.broadcast_to(descs[0].betas[:steps + 1], lnQ.shape)
    return np.stack([beta, lnQ, mbF], -1), np.stack(sums, 1)


def _average(beta, lnQ, mbF, s, R_target, N, weight, q=None, qh=None):
    """The weighted averages of M runs, fields in the order of pa_wavg; s: R_i and
    the moment sums; q: (sum_absq, n_q); qh: overlap histograms."""
    M, n = lnQ.shape
    R = s[..., 0]
    lam = np.log(R) + mbF
    if weight == 0:
        lam[:, 1:] += np.cumsum(np.log(R[:, :-1] / R_target), axis=1)
    w = np.exp(lam - lam.max(0))
    w /= w.sum(0)
    raw = [s[..., 1 + p] / (R * float(N) ** (p % 4 + 1)) for p in range(8)]
    e, e2, e3, e4, m, m2, m3, m4 = raw

    def av(x):
        return (w * x).sum(0)

    We, We2, We3, We4, Wm, Wm2, Wm3, Wm4 = (av(x) for x in raw)

    def central(k, v):
        v = [1.0] + v
        return sum((-1.0) ** (k - l) * math.comb(k, l) * v[1] ** (k - l) * v[l] for l in range(k + 1))

    lnWQ = np.log((w[:, :-1] * np.exp(lnQ[:, 1:] - lnQ[:, 1:].max(0))).sum(0)) + lnQ[:, 1:].max(0)
    WF = N * math.log(2.0) + np.concatenate([[0.0], np.cumsum(lnWQ)])
    zero = np.zeros(n)
    absq = av(q[0] / (N * np.maximum(q[1], 1.0))) if q is not None else zero
    with np.errstate(all="ignore"):
        U4, U4c = 1.0 - Wm4 / (3.0 * Wm2 * Wm2), av(1.0 - m4 / (3.0 * m2 * m2))
    out = np.stack([beta, We, We2, Wm, Wm2, beta**2 * N * (We2 - We * We), beta * N * (Wm2 - Wm * Wm),
                    av(beta**2 * N * (e2 - e * e)), av(beta * N * (m2 - m * m)), WF, absq, zero, w.max(0), w.sum(0),
                    We3, We4, Wm3, Wm4, central(3, [We, We2, We3]), central(4, [We, We2, We3, We4]),
                    central(3, [Wm, Wm2, Wm3]), central(4, [Wm, Wm2, Wm3, Wm4]), U4, U4c, zero], -1)
    if qh is None:
        return out, None
    return out, np.einsum("mi,mid->id", w / np.maximum(q[1], 1.0), qh.astype(np.float64))


def exact(case, seed):
    if case["kind"] == "wavg":
        rec, qh = _host_records(case, seed)
        low = {"sumE3", "sumE4", "sumAbsM3", "sumM4"}
        s = np.stack([rec["R"].astype(np.float64)] +
                     [(rec[f][..., 0].view(np.int64) if f in low else rec[f]).astype(np.float64)
                      for f in ("sumE", "sumE2", "sumE3", "sumE4", "sumAbsM", "sumM2", "sumAbsM3", "sumM4")], -1)
        out, Pq = _average(rec["beta"][0], rec["lnQ"], rec["minus_betaF"], s, case["R"], case["L"] ** 2, case["weight"],
                           (rec["sum_absq"].astype(np.float64), rec["n_q"].astype(np.float64)), qh)
        return {"wavg": out} if Pq is None else {"wavg": out, "Pq": Pq}
    if case["kind"] == "serve" or "," in case["L"] or "," in case["R"] or int(case["L"]) > 32:
        return None
    draws = case["runs"] * int(case["R"]) * case["steps"]
    N = int(case["L"]) ** 2
    if draws * (max(case["theta"] * N, 64)) > 2.5e10 or int(case["R"]) * case["runs"] * N > 3e8 and case["theta"]:
        return None
    descs = _descs(case, seed)
    f, s = _simulate(descs, case["steps"])
    out = {"floats": f if case["read"] == "records" else f[:, -1], "whole": None}
    if case["group"] and case["overlap"] == "none":
        M = case["group"]
        out["wavg"] = np.stack([_average(descs[0].betas, *(x[g:g + M] for x in (f[..., 1], f[..., 2], s)),
                                         int(case["R"]), N, W_FULL)[0] for g in range(0, case["runs"], M)])
    return out
