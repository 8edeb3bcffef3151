"""The calls whose time matters to a user of the simulator, with their inputs and what they return.

Each case is a dict of plain values.  ``prepare`` builds what a user's program holds before the
call (request arrays on the device or on the host, simulator contexts that live across calls),
``run`` makes one pass through the public entry points: for simulations, new requests are loaded
and simulated on every pass, as in ``sweep.py``, ``run.py`` and the benchmark.

Request shapes follow the workloads of ``workloads.py`` (50 requests; 1000 requests with short
prompts; the 2000-request bimodal alpha sweep; 10^4- and 10^5-request Poisson streams; the load
sweep of the paper's Section 6); every seed draws new requests of the same distribution.
"""
import math
from fractions import Fraction

import numpy as np
import torch

import paper_2508_14544_gb300 as G
from paper_2508_14544_gb300 import _lib as L
from paper_2508_14544_gb300 import workloads as W

FIELDS = ("total_latency", "makespan", "peak_memory", "evictions", "steps", "request_steps", "status")
COEF = (12.5, 0.31, 2.7e-5, 0.017, 3.0)  # c0, c1, c2, c3, c_idle of a batch-time model


def listed():
    return [
        # One small instance from host arrays: a what-if query, where call overhead counts.
        dict(name="single_50", kind="sim", source="uniform", policies="A_min", n_inst=1, n=50, ragged=False, M=2000,
             s_max=20, o_max=100, alphas="1/2", host=True, option="", completions=False, batch_time=False, ratio=False),
        # The load sweep of the paper's Section 6: 4 seeds x 10 ragged loads of 200..2000 requests
        # under rough predictions, the three main policies, host arrays (what sweep.py runs).
        dict(name="paper_sweep", kind="sim", source="sweep", intervals="rough", policies="A_max,A_min,H-SF", n_inst=40,
             n=2000, ragged=True, M=10000, host=True, option="", completions=False, batch_time=False, ratio=False),
        # 1024 instances x 1000 requests, four accuracies: a study over seeds on one accelerator
        # that holds all instances at once, where the slowest instance sets the time.
        dict(name="thousand", kind="sim", source="uniform", policies="A_max,A_min", n_inst=1024, n=1000, ragged=False,
             M=16384, s_max=64, o_max=512, alphas="1/5,1/2,4/5,1/1", host=False, option="", completions=False,
             batch_time=False, ratio=False),
        # A tenth of the alpha sweep with the default options: the policies that a study compares
        # besides A_max, and their competitive ratios against hindsight shortest-first.
        dict(name="policy_grid", kind="sim", source="bimodal", policies="A_min,A_ell,A_r,H-SF", n_inst=4096, n=2000,
             ragged=False, M=32768, s_max=256, alphas=",".join(f"{k}/10" for k in range(1, 11)), host=False, option="",
             completions=False, batch_time=False, ratio=True),
        # The whole alpha sweep, the benchmark's step: three policies with the residency tuned on
        # the first run, and the competitive ratios.
        dict(name="alpha_sweep", kind="sim", source="bimodal", policies="A_max,A_min,H-SF", n_inst=40960, n=2000,
             ragged=False, M=32768, s_max=256, alphas=",".join(f"{k}/10" for k in range(1, 11)), host=False,
             option="tune_residency", completions=False, batch_time=False, ratio=True),
        # Ragged instances with the instrumented options of a latency study: batch-time sums, times
        # under a linear model, and every request's completion step.
        dict(name="batch_time", kind="sim", source="uniform", policies="A_max,A_min", n_inst=513, n=777, ragged=True,
             M=12000, s_max=64, o_max=400, alphas="1/4,3/5", host=False, option="", completions=True, batch_time=True,
             ratio=False),
        # Online serving: 256 Poisson streams of 10^4 requests near saturation, with completions.
        dict(name="online_256x1e4", kind="sim", source="lognormal", policies="A_min", n_inst=256, n=10000, ragged=False,
             M=65536, rate=0.5, alphas="3/5", host=False, option="", completions=True, batch_time=False, ratio=False),
        # The longest streams: 64 x 10^5 requests with heavy-tailed lengths.
        dict(name="online_64x1e5", kind="sim", source="zipf", policies="A_max", n_inst=64, n=100000, ragged=False,
             M=500000, rate=2.0, alphas="3/10", host=False, option="", completions=False, batch_time=False, ratio=False),
        # A loop that must not allocate: near the fixed scratch's limit of 262,144 requests.
        dict(name="noalloc", kind="noalloc", policy="A_min", n_inst=250, n=1048, ragged=True, M=8192, s_max=64, o_max=300,
             alphas="1/2"),
        # The analytic ratio of A_min over many short histograms (a scan over predictors) and over
        # a few long ones (lengths up to thousands of tokens).
        dict(name="lemma_many", kind="lemma", n_hist=1 << 20, len=64, l=1, s=0.0),
        dict(name="lemma_long", kind="lemma", n_hist=333, len=1999, l=2, s=41.0),
        # The spectral-radius curve of the corollary, u up to 20,000.
        dict(name="rho_curve", kind="rho", u_max=20000, points=25),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["batch", "batch", "sweep", "online", "noalloc", "lemma", "lemma", "rho"])
    alphas = rng.sample(["1/10", "1/5", "3/10", "1/4", "1/2", "3/5", "4/5", "9/10", "1/1"], rng.randint(1, 4))
    a_min = min(float(Fraction(a)) for a in alphas)
    policies = ",".join(rng.sample(["A_max", "A_min", "H-SF", "A_r", "A_ell"], rng.randint(1, 3)))
    flags = dict(option=rng.choice(["", "", "dense_residency"]), completions=rng.random() < 0.3,
                 batch_time=rng.random() < 0.2)
    if kind == "batch":
        n = _log_int(rng, 20, 2048)
        n_inst = min(_log_int(rng, 1, 8192), 8_000_000 // n)
        s_max, o_max = _log_int(rng, 8, 256), _log_int(rng, 16, 1024)
        M = max(int(s_max + o_max / a_min) + 8, int(rng.uniform(10, 120) * (s_max + o_max) / 2))
        return dict(kind="sim", source="uniform", policies=policies, n_inst=n_inst, n=n, ragged=rng.random() < 0.5, M=M,
                    s_max=s_max, o_max=o_max, alphas=",".join(alphas), host=n * n_inst < 200_000 and rng.random() < 0.5,
                    ratio="H-SF" in policies, **flags)
    if kind == "sweep":
        return dict(kind="sim", source="sweep", intervals=rng.choice(["rough", "buckets", "overlap"]), policies=policies,
                    n_inst=10 * rng.randint(1, 8), n=2000, ragged=True, M=rng.randint(6000, 20000), host=True,
                    ratio="H-SF" in policies, **flags)
    if kind == "online":
        n = _log_int(rng, 300, 30000)
        n_inst = min(_log_int(rng, 1, 512), 2_000_000 // n)
        return dict(kind="sim", source="lognormal", policies=policies, n_inst=n_inst, n=n, ragged=rng.random() < 0.5,
                    M=65536, rate=rng.uniform(0.2, 0.7), alphas=",".join(alphas), host=False, ratio=False, **flags)
    if kind == "noalloc":
        n = _log_int(rng, 10, 2048)
        n_inst = min(_log_int(rng, 1, 8192), 262144 // n)
        s_max, o_max = _log_int(rng, 8, 128), _log_int(rng, 16, 512)
        M = max(int(s_max + o_max / a_min) + 8, int(rng.uniform(10, 100) * (s_max + o_max) / 2))
        return dict(kind="noalloc", policy=rng.choice(["A_max", "A_min", "H-SF"]), n_inst=n_inst, n=n,
                    ragged=rng.random() < 0.5, M=M, s_max=s_max, o_max=o_max, alphas=",".join(alphas))
    if kind == "lemma":
        n_len = _log_int(rng, 2, 8192)
        return dict(kind="lemma", n_hist=min(_log_int(rng, 1, 1 << 20), (1 << 26) // n_len), len=n_len,
                    l=rng.randint(1, 20), s=float(rng.choice([0.0, 0.5, 11.0, 41.0])))
    return dict(kind="rho", u_max=_log_int(rng, 10, 20000), points=_log_int(rng, 1, 40))


# --- inputs ------------------------------------------------------------------------------------------


def _sizes(case):
    """Requests per instance (the same for every seed, as in a study that redraws its requests)."""
    n, k = case["n"], case["n_inst"]
    if not case["ragged"]:
        return np.full(k, n, dtype=np.int64)
    return np.random.default_rng([n, k, 11]).integers(max(1, n // 2), n + 1, size=k, dtype=np.int64)


def _requests(case, seed):
    """Offsets (host) and int32 arrays a, s, l, u, o (device) of independent random instances."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    sizes = _sizes(case)
    off = np.zeros(len(sizes) + 1, dtype=np.int64)
    np.cumsum(sizes, out=off[1:])
    nt = int(off[-1])

    def ints(lo, hi):  # uniform on {lo..hi}
        return torch.randint(lo, hi + 1, (nt,), generator=g, device="cuda", dtype=torch.int64)

    def unif():
        return torch.rand(nt, generator=g, device="cuda", dtype=torch.float64)

    source = case.get("source", "uniform")
    if source == "uniform":
        s, o = ints(1, case["s_max"]), ints(1, case["o_max"])
    elif source == "bimodal":  # 70 % short answers, 30 % long ones
        s = ints(16, case["s_max"])
        o = torch.where(unif() < 0.7, ints(1, 32), ints(512, 2048))
    elif source == "lognormal":
        z = torch.randn(nt, generator=g, device="cuda", dtype=torch.float64)
        s = torch.exp(5.0 + 0.8 * z).round().clamp(1, 4096).long()
        o = torch.ceil(torch.log1p(-unif()) / math.log1p(-1.0 / 300.0)).clamp(1, 4096).long()
    else:  # zipf: exponent 1.2 clipped to 8192 (the clipped mass sits at 8192)
        s = ints(1, 2048)
        cdf = torch.cumsum(torch.arange(1, 8192, device="cuda", dtype=torch.float64) ** -1.2, 0) / 5.591582441177751
        o = (torch.searchsorted(cdf, unif()) + 1).clamp(1, 8192)
    # l ~ U{ceil(alpha o)..o}, u = ceil(l / alpha), in integers; consecutive blocks of instances
    # share an alpha
    fr = [Fraction(a) for a in case["alphas"].split(",")]
    pick = torch.arange(len(sizes), device="cuda") * len(fr) // len(sizes)
    pick = torch.repeat_interleave(pick, torch.from_numpy(sizes).cuda())
    num = torch.tensor([f.numerator for f in fr], device="cuda")[pick]
    den = torch.tensor([f.denominator for f in fr], device="cuda")[pick]
    lo = (num * o + den - 1) // den
    l = lo + ints(0, (1 << 40) - 1) % (o - lo + 1)
    u = (l * den + num - 1) // num
    if "rate" in case:
        c = torch.cumsum(-torch.log1p(-unif()) / case["rate"], 0)
        start = torch.cat([torch.zeros(1, device="cuda", dtype=torch.float64), c])[torch.from_numpy(off[:-1]).cuda()]
        a = (c - torch.repeat_interleave(start, torch.from_numpy(sizes).cuda())).clamp(min=0).floor().long()
    else:
        a = torch.zeros(nt, device="cuda", dtype=torch.int64)
    return off, [x.to(torch.int32).contiguous() for x in (a, s, l, u, o)]


def _sweep_requests(case, seed):
    """Ragged loads of 200..2000 requests, each a random subset of a 2000-request pool."""
    parts = []
    for k in range(case["n_inst"] // 10):
        s_pool, o_pool = W.lookalike_pool(seed * 1000 + k)
        rng = np.random.default_rng([seed, k, 7])
        for n in range(200, 2001, 200):
            pick = rng.choice(s_pool.size, size=n, replace=False)
            s, o = s_pool[pick], o_pool[pick]
            if case["intervals"] == "rough":
                l, u = W.intervals_rough(o)
            elif case["intervals"] == "buckets":
                l, u = W.intervals_buckets(o)
            else:
                l, u = W.intervals_overlap(o, Fraction(19, 20))
            parts.append(dict(a=np.zeros(n, np.int32), s=s, o=o, l=l, u=u))
    w = W.concat_instances("sweep", case["M"], parts)
    w.seed0 = seed
    return w


def _histograms(case, seed):
    """Counts per output length: Poisson counts around a decaying profile, first length present."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    n, m = case["n_hist"], case["len"]
    mean = 40.0 * torch.exp(-3.0 * torch.arange(m, device="cuda", dtype=torch.float64) / m)
    scale = 0.25 + torch.rand(n, 1, generator=g, device="cuda", dtype=torch.float64)
    x = torch.rand(n, m, generator=g, device="cuda", dtype=torch.float64)
    x.mul_(2.0 * mean).mul_(scale).floor_()
    x[:, 0] += 1.0
    return x


def _u_values(case, seed):
    """Increasing u, spaced over the logarithm of 1..u_max with a little jitter, u_max included."""
    r = np.random.default_rng([seed, 5])
    t = (np.arange(case["points"]) + r.random(case["points"])) / case["points"]
    us = np.maximum(1, np.floor(case["u_max"] ** t)).astype(np.int32)
    us[-1] = case["u_max"] - int(r.integers(0, max(1, case["u_max"] // 50)))
    return us


class _Sims:
    """Contexts that live across passes, and the requests in hand."""

    def __init__(self, case, seed):
        self.case = case
        if case["source"] == "sweep":
            self.w = _sweep_requests(case, seed)
            self.off, self.dev = self.w.offsets, None
        else:
            self.off, self.dev = _requests(case, seed)
            if case["host"]:
                a, s, l, u, o = (x.cpu().numpy() for x in self.dev)
                self.w = W.Workload("requests", case["M"], self.off, a, s, l, u, o, seed0=seed)
            else:
                self.w = None
        self.n_total = int(self.off[-1])
        self.rank = None
        names = case["policies"].split(",")
        if "A_r" in names and not case["host"]:
            r = np.random.default_rng([seed, 3])
            self.rank = torch.from_numpy(
                np.concatenate([r.permutation(int(k)) for k in np.diff(self.off)]).astype(np.int32)).cuda()
        elif "A_r" in names:
            self.w.ranks()
        opts = {case["option"]: 1} if case["option"] else {}
        self.sims = {}
        for p in names:
            sim = G.Simulator(G.POLICIES[p], case["M"], case["n_inst"], record_completions=int(case["completions"]),
                              batch_time=int(case["batch_time"]), **opts)
            if not case["host"]:
                sim.set_tie_seeds(np.arange(case["n_inst"], dtype=np.uint64) + np.uint64(seed))
            self.sims[p] = sim


def prepare(case, seed):
    if case["kind"] == "sim":
        return _Sims(case, seed)
    if case["kind"] == "noalloc":
        off, dev = _requests(case, seed)
        out = torch.zeros((case["n_inst"], 7), dtype=torch.int64, device="cuda")
        return dict(case=case, off=off, dev=dev, out=out)
    if case["kind"] == "lemma":
        return dict(case=case, x=_histograms(case, seed))
    return dict(case=case, u=_u_values(case, seed))


# --- one pass ----------------------------------------------------------------------------------------


def run(state):
    if isinstance(state, _Sims):
        return _run_sims(state)
    case = state["case"]
    if case["kind"] == "noalloc":
        rc = L.sim_run_noalloc(G.POLICIES[case["policy"]], case["M"], state["off"], *state["dev"], state["out"])
        if rc != 0:
            raise L.SimError(rc, L.sim_last_error(None))
        return state["out"]
    if case["kind"] == "lemma":
        return G.cr_amin_lemma(state["x"], case["l"], case["s"])
    return G.cr_amin_rho(state["u"])


def _run_sims(st):
    case, out = st.case, {}
    for name, sim in st.sims.items():
        if case["host"]:
            sim.load_workload(st.w)
        else:
            sim.load(st.off, *st.dev, rank=st.rank if name == "A_r" else None)
        res = sim.run()
        for f in FIELDS:
            out[f"{name}.{f}"] = res[f]
        if case["completions"]:
            out[f"{name}.completions"] = sim.completions(st.n_total)
        if case["batch_time"]:
            out[f"{name}.time"] = sim.batch_time(COEF)
            out[f"{name}.sums"] = sim.batch_time_sums()
    if case["ratio"]:
        for name, sim in st.sims.items():
            if name != "H-SF":
                out[f"{name}.ratio"] = sim.competitive_ratio(st.sims["H-SF"])
    return out


# --- what a pass cannot do without, and what its results may differ by ----------------------------------


def work(case):
    if case["kind"] == "lemma":
        n = case["n_hist"] * case["len"]
        # per length: three running sums and their two products (12 flops), read once
        return {"bytes": 8 * n + 8 * case["n_hist"], "flops": 12 * n}
    if case["kind"] == "rho":
        # per iteration and entry: two operator products, a tridiagonal solve step and a scaling
        total = sum(float(x) for x in _u_values(case, 0))
        return {"bytes": 12 * case["points"], "flops": int(30 * 40 * total)}
    n_total = case["n_inst"] * case["n"] * (3 / 4 if case["ragged"] else 1)
    if case["kind"] == "sim" and case["source"] == "sweep":
        n_total = case["n_inst"] * 1100
    pols = 1 if case["kind"] == "noalloc" else len(case["policies"].split(","))
    b = 20 * n_total + pols * 56 * case["n_inst"]
    if case["kind"] == "sim":
        b += pols * (8 * n_total * case["completions"] + 64 * case["n_inst"] * case["batch_time"])
        b += 8 * case["n_inst"] * case["ratio"] * (pols - 1)
        if "A_r" in case["policies"]:
            b += 4 * n_total
    return {"bytes": int(b), "flops": 0}


def tolerance(case):
    if case["kind"] == "lemma":
        return {"rel": 2e-14, "max": 2e-13}  # double-precision running sums of up to 8192 terms
    if case["kind"] == "rho":
        # sums as totals minus prefixes lose digits with u: 6e-9 from the 64-bit value at u = 20,000
        return {"rel": 2.5e-8, "max": 1e-7}
    return "exact"  # integers, and doubles defined as IEEE expressions of integers


def exact(case, seed):
    if case["kind"] == "lemma":
        x = _histograms(case, seed)
        k = case["l"] + torch.arange(case["len"], device="cuda", dtype=torch.float64)
        delta = torch.ones_like(k)
        delta[0] = case["s"] + case["l"]
        out = []
        for xb in torch.split(x, max(1, (1 << 23) // case["len"])):
            def tail(v):  # sums over lengths >= k
                return torch.flip(torch.cumsum(torch.flip(v, [1]), 1), [1])
            f = xb / (case["s"] + k)
            w = tail(f)
            gap = torch.zeros_like(w)
            gap[:, :-1] = tail(w)[:, 1:]  # sum over i > k of (i - k) x_i / (s + i)
            num = (delta * tail(k * xb) * (2.0 * gap + delta * w)).sum(1)
            cnt = tail(xb)
            den = (k * (case["s"] + k) * xb * (2.0 * cnt - xb)).sum(1)
            out.append(num / den)
        return torch.cat(out)
    if case["kind"] == "rho":
        return np.array([_rho(int(u)) for u in _u_values(case, seed)])
    return None  # integer results of a serial simulation: no closed form


def _rho(u):
    """Spectral radius of B^-1 A by power iteration with O(u) products from running sums."""
    i = np.arange(1, u + 1, dtype=np.float64)
    d = np.where(i < u, 4.0 * i / (4.0 * i * i - 1.0), 1.0 / (2.0 * i - 1.0))
    e = 1.0 / (2.0 * i + 1.0)

    def after(v):  # sums over j > i
        return np.concatenate([np.cumsum(v[::-1])[::-1][1:], [0.0]])

    v, lam = np.ones(u), 0.0
    for _ in range(200):
        q2 = np.cumsum(i * i * v)
        r0 = after(v)
        av = 0.5 * i * np.sum(i * v) + q2 - np.cumsum(i ** 3 * v) / (2.0 * i) + i * i * r0 - 0.5 * i ** 3 * after(v / i)
        bv = q2 + i * i * r0
        new = float(v @ av) / float(v @ bv)
        z = d * av
        z[1:] -= av[:-1] * e[:-1]
        z[:-1] -= av[1:] * e[:-1]
        v = z / np.max(np.abs(z))
        if abs(new - lam) <= 1e-15 * new:
            return new
        lam = new
    return lam
