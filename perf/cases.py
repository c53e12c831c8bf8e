"""The work that is measured: population-annealing runs through the public entry points.

A case is a plain dict; `kind` says which program it stands for:

  anneal    one run (paper_2006_00561_gb300.pa.Run): created in the caller's workspace, `steps` steps of
            its schedule of K, the last one streamed out so that the whole final population lands in
            the caller's pinned host buffer, then the records of every step
  adaptive  one run on adaptive temperature steps: the decision, the resample and the sweeps of each
            step by their own calls, then the records and the final population
  batch     many runs advanced together (Batch.run_steps), then every run's records and the energy
            level of each of its replicas
  scan      the copy counts and their scan in the caller's own buffers
            (pa_copy_counts_scan_noalloc)
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_2006_00561_gb300 import pa, workloads

MODELS = {"ferro": pa.MODEL_FERRO, "pmj": pa.MODEL_PMJ}
LAYOUTS = {"packed": pa.LAYOUT_PACKED, "int8": pa.LAYOUT_INT8}
RULES = {"nearest": pa.RESAMPLE_NEAREST, "poisson": pa.RESAMPLE_POISSON,
         "multinomial": pa.RESAMPLE_MULTINOMIAL}
WHOLE = ("step", "R", "sumE", "sumE2", "sumAbsM", "sumM2")
AVERAGES = ("beta", "lnQ", "lnZ", "e", "cv", "m_abs", "chi")
OPS_PER_ATTEMPT = 19.5  # 32-bit integer operations of one Metropolis attempt (Philox4x32-10, test, lattice)


def _anneal(name, dim, L, R0, K, steps, theta, model="ferro", layout="packed", beta0=0.0,
            beta_max=1.0, rule="nearest", heat=False, kind="anneal", target=0.0):
    return dict(name=name, kind=kind, dim=dim, L=L, R0=R0, K=K, steps=steps, theta=theta,
                model=model, layout=layout, beta0=beta0, beta_max=beta_max, rule=rule, heat=heat,
                target=target)


def _batch(name, mix, n, mix_seed, lo, hi, steps, theta=10):
    return dict(name=name, kind="batch", mix=mix, n=n, mix_seed=mix_seed, lo=lo, hi=hi, steps=steps,
                theta=theta)


def listed():
    return [
        # the smallest whole run: byte spins, 1000 replicas, 100 steps; launches and latency
        _anneal("int8_L16_R1000", 2, 16, 1000, 100, 100, 10, layout="int8"),
        # the paper's run on one GPU (L = 64, 20480 replicas, 200 steps) with one sweep per step:
        # the reweight, resample and records weigh as much as the sweeps
        _anneal("L64_R20480_theta1", 2, 64, 20480, 200, 200, 1),
        # the same with ten sweeps per step, a quarter of the schedule
        _anneal("L64_R20480_theta10", 2, 64, 20480, 200, 50, 10),
        # the largest population of the benchmark, first steps of its schedule
        _anneal("L64_R2097152", 2, 64, 1 << 21, 400, 4, 10),
        # the largest lattice: 16385 energy levels, 2 KB per replica, an odd population
        _anneal("L128_R5001", 2, 128, 5001, 200, 20, 10),
        # one spin-glass instance of the disorder ensemble, alone
        _anneal("ea3d_L10_R16384", 3, 10, 1 << 14, 150, 40, 10, model="pmj", beta_max=3.0),
        # the smallest spin-glass request: a few thousand replicas, ragged
        _anneal("ea3d_L6_R4099", 3, 6, 4099, 100, 60, 10, model="pmj", beta_max=3.0),
        # heating from the ground state on adaptive steps, with the paper's Poisson copies
        _anneal("adaptive_heating_L32", 2, 32, 20000, 64, 16, 5, beta0=1.0, beta_max=0.0,
                rule="poisson", heat=True, kind="adaptive", target=0.85),
        # multinomial copies of a large population, one sweep per step: the resample weighs
        _anneal("multinomial_L32_R150001", 2, 32, 150001, 100, 30, 1, rule="multinomial"),
        # a disorder ensemble of spin glasses advanced together
        _batch("ensemble_ea3d", "ea", 24, 4, 12, 14, 30),
        # a serving batch: lattices of every class, requests from 2^8 to 2^14 replicas
        _batch("serving_mix", "serving", 28, 5, 8, 14, 25),
        # copy counts and scan for callers that cannot allocate
        dict(name="scan_R3000017", kind="scan", R=3000017, bins=4097),
    ]


BUDGET = 3.0e11  # attempts of a drawn pass (the largest listed case makes 3.4e11)


def _fit(rng, per_step, top):
    """Steps that keep a pass under the budget, at least 4."""
    most = max(4, int(BUDGET / max(per_step, 1)))
    return max(4, min(top, most, int(math.exp(rng.uniform(math.log(8), math.log(201))))))


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["anneal"] * 5 + ["adaptive", "batch", "batch", "scan"])
    if kind == "scan":
        return dict(kind="scan", R=_log_int(rng, 1000, pa.NOALLOC_MAX_REPLICAS),
                    bins=rng.choice([129, 301, 769, 1501, 4097, 16385]))
    if kind == "batch":
        mix = rng.choice(["ea", "serving"])
        lo = rng.randint(8, 12)
        case = _batch("", mix, rng.randint(4, 28), rng.randint(1, 10 ** 6), lo,
                      lo + rng.randint(0, 2), rng.randint(8, 40), rng.choice([1, 5, 10]))
        case.pop("name")
        return case
    dim = rng.choice([2, 2, 3])
    L = rng.choice([8, 16, 32, 64, 128] if dim == 2 else [4, 6, 8, 10, 12, 16])
    model = "pmj" if dim == 3 else rng.choice(["ferro", "ferro", "pmj"])
    layout = rng.choice(["packed", "packed", "int8"]) if L <= 64 else "packed"
    theta = rng.choice([1, 2, 5, 10, 20])
    N = L ** dim
    # up to a gigabyte of spins and to 2^20 replicas, a sixteenth of that as bytes
    most = min(1 << 20, (1 << 33) // N) // (16 if layout == "int8" else 1)
    R0 = _log_int(rng, 300, max(600, most))
    rule = rng.choice(["nearest", "nearest", "poisson", "multinomial"])
    heat = model == "ferro" and rng.random() < 0.25
    beta = rng.choice([0.6, 1.0] if heat else [0.5, 1.0, 2.0] if dim == 2 else [1.0, 3.0])
    K = rng.randint(60, 300)
    steps = min(K, _fit(rng, 20 * R0 * N * theta, K))
    if kind == "adaptive":
        steps = min(steps, 24)
    case = _anneal("", dim, L, R0, K, steps, theta, model, layout, beta if heat else 0.0,
                   0.0 if heat else beta, rule, heat, kind, 0.85 if kind == "adaptive" else 0.0)
    case.pop("name")
    return case


# ---- what a user's program has in hand ---------------------------------------
def _config(case, rng):
    return pa.make_config(
        dim=case["dim"], L=case["L"], model=MODELS[case["model"]], layout=LAYOUTS[case["layout"]],
        K=case["K"], theta=case["theta"], instance_id=rng.randrange(1 << 20), R0=case["R0"],
        beta0=case["beta0"], beta_max=case["beta_max"], seed=rng.randrange(1, 1 << 63),
        coupling_seed=rng.randrange(1, 1 << 63) if case["model"] == "pmj" else 0,
        init=pa.INIT_GROUND if case["heat"] else pa.INIT_RANDOM, resample=RULES[case["rule"]])


def _mix(case, rng):
    """The runs of a batch: sizes and schedules of the workload generators, fresh random streams."""
    if case["mix"] == "ea":
        specs = workloads.ea_ensemble(case["n"], seed=case["mix_seed"], theta=case["theta"],
                                      R0s=tuple(1 << e for e in range(case["lo"], case["hi"] + 1)))
    else:
        specs = workloads.serving_trace(case["n"], seed=case["mix_seed"], theta=case["theta"],
                                        R0_exp=(case["lo"], case["hi"]))
    out = []
    for s in specs:
        s = {k: v for k, v in s.items() if k != "arrival"}
        s.update(seed=rng.randrange(1, 1 << 63), coupling_seed=rng.randrange(1, 1 << 63))
        out.append(pa.make_config(**s))
    return out


def _scan_inputs(case, seed):
    """Energy levels of a population around its mean and the copy tables of a small step."""
    r = np.random.default_rng(seed)
    bins = case["bins"]
    width = max(2.0, math.sqrt(bins) / 2)
    ebin = np.clip(np.rint(r.normal(0.3 * bins, width, case["R"])), 0, bins - 1).astype(np.int32)
    k = np.arange(bins)
    tau = np.minimum(np.exp(-(k - ebin.mean()) * (0.3 / width)), 50.0)
    n = np.floor(tau)
    F = np.floor((tau - n) * 2.0 ** 32).astype(np.uint32).view(np.int32)
    return ebin, n.astype(np.int32), F


def _stride(cfg):
    if cfg.layout == pa.LAYOUT_PACKED:
        return (cfg.L ** (cfg.dim - 1) * ((cfg.L + 31) // 32) * 4 + 15) // 16 * 16
    return (cfg.L ** cfg.dim + 15) // 16 * 16


def _capacity(cfg):
    return cfg.R0 + 16 * math.ceil(math.sqrt(cfg.R0)) + 1024


def prepare(case, seed):
    rng = random.Random(seed)
    st = {"case": case, "stream": torch.cuda.current_stream()}
    if case["kind"] == "scan":
        ebin, n, F = (torch.from_numpy(a).cuda() for a in _scan_inputs(case, seed))
        st.update(ebin=ebin, n=n, F=F, seed=rng.randrange(1, 1 << 63), step=rng.randrange(1, 200),
                  instance=rng.randrange(1 << 20), counts=torch.empty_like(ebin),
                  offsets=torch.empty_like(ebin), total=torch.empty(1, dtype=torch.int32, device="cuda"))
        return st
    cfgs = _mix(case, rng) if case["kind"] == "batch" else [_config(case, rng)]
    st["cfgs"] = cfgs
    st["ws"] = [torch.empty(pa.pa_workspace_size(c), dtype=torch.uint8, device="cuda") for c in cfgs]
    if case["kind"] == "anneal":
        st["host"] = torch.zeros(_capacity(cfgs[0]) * _stride(cfgs[0]), dtype=torch.uint8,
                                 pin_memory=True)
        st["copies"] = torch.cuda.Stream()
    elif case["kind"] == "adaptive":
        st["host"] = np.zeros(_capacity(cfgs[0]) * _stride(cfgs[0]), dtype=np.uint8)
    else:
        st["levels"] = np.zeros(sum(_capacity(c) for c in cfgs), dtype=np.int32)
    return st


def _records(run, n):
    rec = run.history(0, n)
    return (np.array([[r[k] for k in WHOLE] for r in rec], dtype=np.int64),
            np.array([[r[k] for k in AVERAGES] for r in rec], dtype=np.float64))


def run(st):
    case = st["case"]
    if case["kind"] == "scan":
        pa.pa_copy_counts_scan_noalloc(
            st["ebin"].data_ptr(), case["R"], st["n"].data_ptr(), st["F"].data_ptr(), case["bins"],
            st["seed"], st["step"], st["instance"], st["counts"].data_ptr(),
            st["offsets"].data_ptr(), st["total"].data_ptr(), st["stream"].cuda_stream)
        return {"counts": st["counts"], "offsets": st["offsets"], "total": st["total"]}
    runs = [pa.Run(c, stream=st["stream"], workspace=w) for c, w in zip(st["cfgs"], st["ws"])]
    n = case["steps"]
    if case["kind"] == "batch":
        batch = pa.Batch(runs, stream=st["stream"])
        batch.run_steps(n)
        assert batch.sync() == pa.PA_OK
        recs = [_records(r, n + 1) for r in runs]
        at = 0
        for r in runs:  # every run's levels at the start of its share of the caller's buffer
            levels = r.dump(pa.DUMP_EBIN)
            st["levels"][at:at + levels.size] = levels.view(np.int32)
            at += _capacity(r.cfg)
        batch.close()
        for r in runs:
            r.close()
        return {"whole": np.concatenate([r[0] for r in recs]),
                "averages": np.concatenate([r[1] for r in recs]), "levels": st["levels"]}
    r = runs[0]
    if case["kind"] == "anneal":
        r.run_steps(n - 1)
        # large populations leave the device range by range while the later ranges sweep
        r.step_stream(st["host"], 8 if st["host"].numel() > (1 << 24) else 1, st["copies"])
        whole, averages = _records(r, n + 1)
    else:
        r.sweep(case["theta"])  # equilibrated at beta0, so that the first decision has a histogram
        for _ in range(n):
            r.resample_to(r.adaptive_beta(case["target"], case["beta_max"]))
            r.sweep(case["theta"])
        whole, averages = _records(r, n + 1)
        spins = r.dump(pa.DUMP_SPINS_RAW)
        st["host"][:spins.size] = spins
    r.close()
    # the caller's buffer holds a full capacity; the population is its first R replicas
    return {"whole": whole, "averages": averages, "population": st["host"]}


def work(case):
    """Populations, levels and magnetisations in and out once per pass; integer operations as flops."""
    if case["kind"] == "scan":
        return {"bytes": 12 * case["R"] + 8 * case["bins"], "flops": 15 * case["R"]}
    cfgs = _mix(case, random.Random(0)) if case["kind"] == "batch" else [_config(case, random.Random(0))]
    n = case["steps"]
    attempts = sum(c.R0 * c.L ** c.dim * c.theta for c in cfgs) * n
    # per step: levels read, counts and offsets written, a replica's spins, level and
    # magnetisation read and written by its resample
    moved = sum(c.R0 * (12 + 2 * (_stride(c) + 8)) for c in cfgs) * n
    return {"bytes": moved, "flops": OPS_PER_ATTEMPT * attempts}


# ---- the same runs in plain torch and numpy ----------------------------------
M32 = 0xFFFFFFFF
INIT, SWEEP, RESAMPLE, COUPLING, POISSON, MULTINOMIAL = 1, 2, 3, 4, 5, 6
EXACT_MOST = 7.0e10  # attempts beyond which exact() takes too long


def _philox(c, key):
    """Philox4x32-10 of int64 tensors of 32-bit words that broadcast together."""
    c0, c1, c2, c3 = torch.broadcast_tensors(*c)
    k0, k1 = key & M32, key >> 32
    for _ in range(10):
        a, b = c0 * 0xD2511F53, c2 * 0xCD9E8D57
        c0, c1, c2, c3 = (((b >> 32) & M32) ^ c1 ^ k0, b & M32, ((a >> 32) & M32) ^ c3 ^ k1, a & M32)
        k0, k1 = (k0 + 0x9E3779B9) & M32, (k1 + 0xBB67AE85) & M32
    return torch.stack((c0, c1, c2, c3), -1)


def _threshold(beta, dE):
    return math.floor(math.exp(-(beta * dE)) * 4294967296.0)


def _poisson1():
    out, p, acc, m = [], math.exp(-1.0), 0.0, 0
    while True:
        acc += p
        v = math.floor(math.ldexp(acc, 32))
        out.append(min(v, M32))
        if v >= M32:
            return out
        m += 1
        p /= m


class _Sim:
    """One run, replica by replica in integers, its weights and averages in float64."""

    def __init__(self, cfg):
        self.c, self.N = cfg, cfg.L ** cfg.dim
        self.dev = "cuda" if torch.cuda.is_available() else "cpu"
        self.shape = (cfg.L,) * cfg.dim
        N, L, dim = self.N, cfg.L, cfg.dim
        self.R, self.g, self.step = cfg.R0, 0, 0
        self.beta, self.lnQ = cfg.beta0, 0.0
        self.bins = dim * N // 2 + 1
        t = lambda *v: [torch.as_tensor(x, dtype=torch.int64, device=self.dev) for x in v]  # noqa: E731
        self.t = t
        q = torch.arange(N // 4, device=self.dev)
        if cfg.init == pa.INIT_GROUND:
            self.s = torch.ones((self.R,) + self.shape, dtype=torch.int8, device=self.dev)
            self.lnZ = math.log(2.0) + cfg.beta0 * dim * N
        else:
            self.s = torch.empty((self.R,) + self.shape, dtype=torch.int8, device=self.dev)
            for lo, hi in self.chunks():
                slot = torch.arange(lo, hi, device=self.dev)[:, None]
                w = _philox(t(q[None], 0, slot, INIT << 28 | cfg.instance_id), cfg.seed)
                self.s[lo:hi] = (1 - 2 * (w >> 31)).to(torch.int8).reshape((hi - lo,) + self.shape)
            self.lnZ = N * math.log(2.0)
        self.J, self.parity = None, 0
        if cfg.model == pa.MODEL_PMJ:
            d = torch.arange(dim, device=self.dev)[:, None]
            w = _philox(t(q[None], d, 0, COUPLING << 28 | cfg.instance_id), cfg.coupling_seed)
            self.J = (1 - 2 * (w >> 31)).to(torch.int8).reshape((dim,) + self.shape)
            self.parity = int((self.J < 0).sum()) & 1
        # colour-c site of pair h: the pair's member whose coordinate sum has that parity
        h = torch.arange(N // 2, device=self.dev)
        row = 2 * h // L
        par = (row & 1) if dim == 2 else ((row % L + row // L) & 1)
        self.site = [row * L + (2 * h) % L + ((c + par) & 1) for c in (0, 1)]
        self.measure()

    def chunks(self):
        per = max(1, (1 << 25) // self.N)
        return [(a, min(self.R, a + per)) for a in range(0, self.R, per)]

    def axis(self, d):  # x is the fastest axis
        return self.c.dim - d

    def measure(self):
        self.level = torch.empty(self.R, dtype=torch.int64, device=self.dev)
        self.mag = torch.empty(self.R, dtype=torch.int64, device=self.dev)
        for lo, hi in self.chunks():
            s = self.s[lo:hi]
            U = 0
            for d in range(self.c.dim):
                b = s * torch.roll(s, -1, self.axis(d))
                b = b if self.J is None else b * self.J[d]
                U = U + (b < 0).reshape(hi - lo, -1).sum(1)
            self.level[lo:hi] = U >> 1
            self.mag[lo:hi] = s.reshape(hi - lo, -1).sum(1, dtype=torch.int64)

    def sweeps(self, n):
        T = torch.tensor([0, 0, 0, 0], device=self.dev)
        T[0] = 1 << 33  # dE <= 0
        for k in range(1, 4):
            T[k] = _threshold(self.beta, 4 * k)
        q = torch.arange(self.N // 8, device=self.dev)[None]
        ctag = SWEEP << 28 | self.c.instance_id
        for lo, hi in self.chunks():
            s = self.s[lo:hi].clone()
            slot = torch.arange(lo, hi, device=self.dev)[:, None]
            for t in range(n):
                for c in (0, 1):
                    u = _philox(self.t(2 * (self.g + t) + c, q, ctag, slot), self.c.seed)
                    f = torch.zeros_like(s)
                    for d in range(self.c.dim):
                        a = self.axis(d)
                        if self.J is None:
                            f += torch.roll(s, -1, a) + torch.roll(s, 1, a)
                        else:
                            f += torch.roll(s, -1, a) * self.J[d] + torch.roll(s * self.J[d], 1, a)
                    flat = s.reshape(hi - lo, -1)
                    own = flat[:, self.site[c]]
                    half = own * f.reshape(hi - lo, -1)[:, self.site[c]]  # dE / 2, even
                    ok = u.reshape(hi - lo, -1) < T[(half.clamp(min=0) >> 1).long()]
                    flat[:, self.site[c]] = torch.where(ok, -own, own)
            self.s[lo:hi] = s
        self.g += n
        self.measure()

    def hist(self):
        return torch.bincount(self.level, minlength=self.bins).cpu().numpy().astype(np.float64)

    def overlap(self, db):
        k = np.flatnonzero(self.H)
        j = (k[-1] - k) if db < 0 else (k - k[0])
        w = np.array([math.exp(-(abs(db) * float(4 * x))) for x in j])
        hw = self.H[k] * w
        return np.cumsum(np.minimum(self.H[k] / self.R, hw / np.cumsum(hw)[-1]))[-1]

    def adaptive(self, target, end):
        self.H = self.hist()
        span = end - self.beta
        if span == 0.0 or self.overlap(span) >= target:
            return end
        lo, hi, sgn = 0.0, abs(span), -1.0 if span < 0 else 1.0
        for _ in range(60):
            mid = lo + (hi - lo) * 0.5
            lo, hi = (mid, hi) if self.overlap(sgn * mid) >= target else (lo, mid)
        return self.beta + sgn * lo

    def resample(self, beta):
        c, db, H = self.c, beta - self.beta, self.hist()
        k = np.flatnonzero(H)
        kref = int(k[-1] if db < 0 else k[0])
        j = (kref - k) if db < 0 else (k - kref)
        D = np.array([math.exp(-(abs(db) * float(4 * x))) for x in j])
        S = float(np.sum(H[k] * D))
        tau = np.zeros(self.bins)
        tau[k] = c.R0 * D / S
        n, F = np.floor(tau), np.floor((tau - np.floor(tau)) * 4294967296.0)
        Eref = 2 * (2 * kref + self.parity) - c.dim * self.N
        self.lnQ = math.log(S) - math.log(self.R) - db * Eref
        self.lnZ += self.lnQ
        self.beta, self.step = beta, self.step + 1
        n = torch.from_numpy(n.astype(np.int64)).to(self.dev)[self.level]
        F = torch.from_numpy(F.astype(np.int64)).to(self.dev)[self.level]
        if c.resample == pa.RESAMPLE_NEAREST:
            i = torch.arange((self.R + 3) // 4, device=self.dev)
            u = _philox(self.t(i, self.step, 0, RESAMPLE << 28 | c.instance_id), c.seed)
            r = n + (u.reshape(-1)[:self.R] < F)
        elif c.resample == pa.RESAMPLE_POISSON:
            r = self.poisson(n, F)
        else:
            C = np.cumsum((n << 32).cpu().numpy() + F.cpu().numpy())
            i = torch.arange((c.R0 + 1) // 2, device=self.dev)
            w = _philox(self.t(i, self.step, 0, MULTINOMIAL << 28 | c.instance_id), c.seed)
            v = w.reshape(-1, 2)[:c.R0].cpu().numpy()
            tot = int(C[-1])
            x = np.array([((int(b) << 32 | int(a)) * tot) >> 64 for a, b in v], dtype=np.int64)
            r = torch.from_numpy(np.bincount(np.searchsorted(C, x, "right"), minlength=self.R)).to(self.dev)
        src = torch.repeat_interleave(torch.arange(self.R, device=self.dev), r)
        self.s, self.R = self.s[src], int(src.numel())

    def poisson(self, n, F):
        P1 = torch.tensor(_poisson1(), device=self.dev)
        i = torch.arange(self.R, device=self.dev)

        def word(pos):
            w = _philox(self.t(i, self.step, pos >> 2, POISSON << 28 | self.c.instance_id), self.c.seed)
            return w.gather(1, (pos & 3)[:, None])[:, 0]

        def unit(pos):
            return torch.searchsorted(P1, word(pos), right=True)

        pos = torch.zeros_like(i)
        ev, count = unit(pos), torch.zeros_like(i)
        pos = pos + 1
        for e in range(int(ev.max())):
            count += (e < ev) & (word(pos + e) < F)
        pos = pos + ev
        for j in range(int(n.max())):
            count += torch.where(j < n, unit(pos + j), 0)
        return count

    def averages(self):
        E = 2 * (2 * self.level + self.parity) - self.c.dim * self.N
        R, N, b = float(self.R), float(self.N), self.beta
        mE, mE2 = int(E.sum()) / R, int((E * E).sum()) / R
        mA, mM2 = int(self.mag.abs().sum()) / R, int((self.mag * self.mag).sum()) / R
        return [b, self.lnQ, self.lnZ, mE / N, b * b * (mE2 - mE * mE) / N, mA / N, b * (mM2 - mA * mA) / N]


def exact(case, seed):
    """The averages of every step; the other outputs are whole numbers and bytes."""
    if case["kind"] == "scan" or work(case)["flops"] / OPS_PER_ATTEMPT > EXACT_MOST:
        return None
    rng = random.Random(seed)
    rows = []
    for cfg in _mix(case, rng) if case["kind"] == "batch" else [_config(case, rng)]:
        sim = _Sim(cfg)
        if case["kind"] == "adaptive":
            sim.sweeps(cfg.theta)
        rows.append(sim.averages())
        for i in range(1, case["steps"] + 1):
            if case["kind"] == "adaptive":
                b = sim.adaptive(case["target"], cfg.beta_max)
            else:
                b = cfg.beta0 + ((cfg.beta_max - cfg.beta0) * i) / cfg.K
            sim.resample(b)
            sim.sweeps(cfg.theta)
            rows.append(sim.averages())
    return {"whole": None, "averages": np.array(rows), "population": None, "levels": None}
