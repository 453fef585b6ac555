"""The measured cases: what a user of the nested MLMC library has it do.

Every case goes through the package's public entry points (single levels,
work lists, plans, adaptive estimates, batches, error-model statistics) at
sizes of the benchmark's configurations: levels 0..10, 10^3 samples to 10^8,
the benchmark's market parameters and option ranges.

    listed()             the cases
    draw(rng)            one more case of the same ranges
    prepare(case, seed)  inputs and handles a user's program holds
    run(state)           one pass; the results as the library returns them
    work(case)           algorithmic bytes and operations of a pass
    exact(case, seed)    the results in 64 bits, in plain torch
"""
import math

import numpy as np
import torch

from paper_2502_07123_gb300 import mlmc as m
from paper_2502_07123_gb300 import workloads as W

VARIANTS = {"fp64": m.FP64_EXACT, "fp32": m.FP32_EXACT, "fixed": m.FIXED_APPROX, "fp16": m.FP16_APPROX,
            "bf16": m.BF16_APPROX, "fp16s": m.FP16S_APPROX, "bf16s": m.BF16S_APPROX,
            "corr_fixed": m.NESTED_CORR_FIXED, "corr_fp16": m.NESTED_CORR_FP16, "corr_bf16s": m.NESTED_CORR_BF16S}
APPROX = ("fixed", "fp16", "bf16", "fp16s", "bf16s")
PAYOFFS = {"euro": W.EURO, "digital": W.DIGITAL, "asian": W.ASIAN, "lookback": W.LOOKBACK}
SCHEMES = {"euler": W.EULER, "milstein": W.MILSTEIN}
MODES = {"fp32": m.MODE_PLAIN_FP32, "nested": m.MODE_NESTED_FIXED, "nested_exact_low": m.MODE_NESTED_FIXED_EXACT_LOW,
         "nested_fp16s": m.MODE_NESTED_FP16S}


def _level(name, variant, level, N, payoff="euro", scheme="euler", sigma=0.2, d=10, method=1, pack=0):
    return dict(name=name, kind="level", variant=variant, level=level, N=N, payoff=payoff, scheme=scheme, sigma=sigma,
                d=d, method=method, pack=pack)


def listed():
    return [
        # the smallest call: one correction term of an adaptive loop's first round
        _level("corr_small", "corr_fixed", 3, 1000),
        # plain FP64 MLMC, levels 0..5 with 10^4 samples each, as one work list
        dict(name="fp64_list", kind="list", work="fp64", levels=6, top=10_000, floor=10_000),
        # the nested workload: European and digital call, levels 0..8, packed draws
        dict(name="nested_list", kind="list", work="nested", levels=9, top=10_000_000, floor=10_000),
        # plain FP32 Milstein MLMC over all levels as a resident plan, launched and read
        dict(name="fp32_plan", kind="plan", work="fp32", levels=9, top=16_000_001, floor=10_000, payoff="lookback",
             scheme="milstein"),
        # a low level's approximate term, where most samples are
        _level("approx_low", "fixed", 1, 100_000_007, payoff="digital", pack=1),
        # the throughput sweep's half-precision point: deep, path-dependent
        _level("half_deep", "fp16", 8, 1_000_003, payoff="asian", scheme="milstein"),
        # correction terms: the nested estimator's expensive half
        _level("corr_euro", "corr_fixed", 4, 8_000_009, sigma=0.4),
        _level("corr_asian", "corr_fixed", 7, 1_000_003, payoff="asian", scheme="milstein"),
        # the sweep's FP64 reference estimator
        _level("fp64_level", "fp64", 5, 500_003, scheme="milstein"),
        # time to accuracy: the adaptive nested estimator, every level sampled
        dict(name="estimate", kind="estimate", mode="nested", eps=1e-3, payoff="euro"),
        # many options in one launch (the batched workload, in small)
        dict(name="batch", kind="batch", mode="nested_exact_low", n=24, eps_lo=1e-3, eps_hi=1e-2),
        # error-model statistics for the bit-width optimiser
        dict(name="sensitivities", kind="sens", level=6, N=100_001),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["level"] * 7 + ["list", "plan", "estimate", "batch", "sens"])
    if kind == "level":
        variant = rng.choice(["fp64", "fp32", "fp32", "fixed", "fixed", "corr_fixed", "corr_fixed", "fp16", "bf16",
                              "fp16s", "bf16s", "corr_fp16", "corr_bf16s"])
        level = rng.randrange(11)
        steps = _log(rng, 1e3, 3e7 if variant == "fp64" else 2.5e8)
        d = rng.choice([8, 9, 10, 10, 12])
        pack = rng.randrange(2) if variant in APPROX and d in (9, 10) else 0
        return dict(kind="level", variant=variant, level=level, N=max(37, int(steps) >> level),
                    payoff=rng.choice(list(PAYOFFS)), scheme=rng.choice(list(SCHEMES)),
                    sigma=rng.choice([0.1, 0.2, 0.4]), d=d, method=rng.choice([1, 1, 1, 3]), pack=pack)
    if kind == "list":
        work = rng.choice(["fp64", "nested"])
        return dict(kind="list", work=work, levels=rng.randrange(3, 10),
                    top=int(_log(rng, 1e4, 2e5 if work == "fp64" else 1e7)), floor=rng.randrange(1000, 10_001))
    if kind == "plan":
        return dict(kind="plan", work="fp32", levels=rng.randrange(3, 10), top=int(_log(rng, 2e4, 1.6e7)),
                    floor=rng.randrange(1000, 10_001), payoff=rng.choice(list(PAYOFFS)),
                    scheme=rng.choice(list(SCHEMES)))
    if kind == "estimate":
        return dict(kind="estimate", mode=rng.choice(list(MODES)), eps=_log(rng, 1e-3, 2e-2),
                    payoff=rng.choice(["euro", "digital", "asian"]))
    if kind == "batch":
        return dict(kind="batch", mode=rng.choice(["nested", "nested_exact_low"]), n=rng.randrange(2, 20),
                    eps_lo=2e-3, eps_hi=1e-2)
    level = rng.randrange(11)
    return dict(kind="sens", level=level, N=max(101, int(_log(rng, 1e4, 8e6)) >> level))


# --------------------------------------------------------------------------
# inputs
# --------------------------------------------------------------------------
def _market(seed, **over):
    """The test case's option with spot and strike of the batched workload's range, near the money."""
    rng = np.random.default_rng(seed)
    return W.params(S0=float(rng.uniform(95, 105)), K=float(rng.uniform(95, 105)), **over), int(rng.integers(1 << 62))


def _counts(case):
    return [max(case["floor"], int(case["top"] * 2.0 ** (-1.5 * lev))) for lev in range(case["levels"])]


def _items(case, seed):
    """(market, variant, level, N, request, pack) per item of a list or plan."""
    if case["work"] == "nested":
        out, key = [], 0
        for pay in (W.EURO, W.DIGITAL):
            p, key = _market(seed, payoff=pay)
            for lev, n in enumerate(_counts(case)):
                out += [(p, "fixed", lev, n, pay, 1), (p, "corr_fixed", lev, case["floor"], pay, 1)]
        return out, key
    p, key = _market(seed, payoff=PAYOFFS[case.get("payoff", "euro")], scheme=SCHEMES[case.get("scheme", "euler")])
    return [(p, case["work"], lev, n, 0, 0) for lev, n in enumerate(_counts(case))], key


def _of_level(case, seed):
    return _market(seed, payoff=PAYOFFS[case["payoff"]], scheme=SCHEMES[case["scheme"]], sigma=case["sigma"])


def prepare(case, seed):
    kind = case["kind"]
    if kind == "level":
        p, key = _of_level(case, seed)
        P = m.make_params(p, d=case["d"], method=case["method"], rng_pack=case["pack"])
        return dict(kind=kind, args=(case["level"], case["N"], P, VARIANTS[case["variant"]], key))
    if kind in ("list", "plan"):
        items, key = _items(case, seed)
        works = [dict(params=m.make_params(p, request=req, rng_pack=pack), level=lev, variant=VARIANTS[v], N=n)
                 for p, v, lev, n, req, pack in items]
        if kind == "list":
            return dict(kind=kind, work=m.WorkList(works), key=key)
        return dict(kind=kind, plan=m.Plan(works, key))
    if kind == "estimate":
        p, key = _market(seed, payoff=PAYOFFS[case["payoff"]])
        return dict(kind=kind, args=(case["eps"], m.make_params(p, rng_pack=1), MODES[case["mode"]], key))
    if kind == "batch":
        opts = W.batched_options(case["n"], seed % (1 << 31), (case["eps_lo"], case["eps_hi"]))
        plist = [m.make_params(o, request=i, rng_pack=1) for i, o in enumerate(opts)]
        return dict(kind=kind, args=(plist, [o["eps"] for o in opts], MODES[case["mode"]], seed))
    p, key = _market(seed)
    return dict(kind=kind, args=(case["level"], case["N"], m.make_params(p), key))


# --------------------------------------------------------------------------
# one pass
# --------------------------------------------------------------------------
def _words(lo, hi):
    """The 128-bit sum of squares as 64-bit words."""
    return np.array([lo, hi], dtype=np.uint64).view(np.int64)


def _of_array(a):
    out = {k: a[k] for k in ("sum", "sum2", "isum")}
    out.update({k: a[k].astype(np.uint64).view(np.int64) for k in ("n", "saturations", "isum2_lo", "isum2_hi")})
    return out


def run(state):
    kind = state["kind"]
    if kind == "level":
        r = m.mlmc_level(*state["args"])
        return dict({k: r[k] for k in ("sum", "sum2", "n", "saturations", "isum")},
                    isum2=_words(r["isum2_lo"], r["isum2_hi"]))
    if kind == "list":
        return _of_array(m.mlmc_run(state["work"], state["key"], raw=True))
    if kind == "plan":
        state["plan"].launch()
        return _of_array(state["plan"].results(raw=True))
    if kind == "estimate":
        r = m.mlmc_estimate(*state["args"], max_level=10)
        n = np.zeros((11, 2), dtype=np.int64)   # N by level and estimator, zero above the final level
        n[:r["L"] + 1] = r["N"]
        return dict(r, N=n)
    if kind == "batch":
        r = m.mlmc_batch_estimate(*state["args"], max_level=12, iters_per_launch=-4096)
        return dict(price=np.array(r["price"]), stderr=np.array(r["stderr"]), L=np.array(r["L"]))
    r = m.mlmc_sensitivities(*state["args"], per_instance=True)
    return {k: r[k] for k in ("A", "B", "maxabs", "mean", "var", "n", "inst")}


# --------------------------------------------------------------------------
# the work a pass cannot do without
# --------------------------------------------------------------------------
#: 32-bit operations per fine path-step: Philox 10, the inverse Normal 20, table index 5, an Algorithm-1 step 10
#: and half its coarse one 5.5, an exact step 2 and half its coarse one 1.5
OPS = {"fp64": 33.5, "fp32": 33.5, "approx": 30.5, "corr": 54.0}


def _ops(variant):
    return OPS.get(variant, OPS["approx"] if variant in APPROX else OPS["corr"])


def work(case):
    kind = case["kind"]
    if kind == "level":
        return dict(bytes=536 + 72, flops=_ops(case["variant"]) * (case["N"] << case["level"]))
    if kind in ("list", "plan"):
        items, _ = _items(case, 1)
        return dict(bytes=608 * len(items), flops=sum(_ops(v) * (n << lev) for _, v, lev, n, _, _ in items))
    if kind == "estimate":   # about 300 eps^-2 path-steps to the test case's accuracy
        return dict(bytes=608, flops=OPS["approx"] * 300 / case["eps"] ** 2)
    if kind == "batch":      # the mean of eps^-2 over the log-uniform accuracies
        lo, hi = case["eps_lo"], case["eps_hi"]
        return dict(bytes=608 * case["n"],
                    flops=OPS["approx"] * 600 * case["n"] * (lo ** -2 - hi ** -2) / (2 * math.log(hi / lo)))
    return dict(bytes=608 + 7 * 8 * 3 * (1 << case["level"]) // 2, flops=60.0 * (case["N"] << case["level"]))


# --------------------------------------------------------------------------
# the results in 64 bits
# --------------------------------------------------------------------------
def _mulhilo(a, x):
    lo = (a * x) & 0xFFFFFFFF
    hi = (a * (x >> 16) + ((a * (x & 0xFFFF)) >> 16)) >> 16
    return hi, lo


def _philox(q, ctr2, ctr3, seed):
    """Philox4x32-10 (Salmon et al. 2011) of the counters (q, ctr2, ctr3)."""
    x0, x1, x2, x3 = q & 0xFFFFFFFF, q >> 32, torch.full_like(q, ctr2), torch.full_like(q, ctr3)
    k0, k1 = seed & 0xFFFFFFFF, seed >> 32
    for _ in range(10):
        h0, l0 = _mulhilo(0xD2511F53, x0)
        h1, l1 = _mulhilo(0xCD9E8D57, x2)
        x0, x1, x2, x3 = h1 ^ x1 ^ k0, l1, h0 ^ x3 ^ k1, l0
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    return x0, x1, x2, x3


def _uniforms(s, level, seed, request=0):
    """J of steps 0, 1, ... of the samples s (stream 0)."""
    if level >= 2:
        for c in range(1 << (level - 2)):
            yield from _philox((s << (level - 2)) + c, level, request, seed)
    else:
        for i in range(1 << level):
            w = (s << level) + i
            x = torch.stack(_philox(w >> 2, level, request, seed))
            yield x.gather(0, (w & 3)[None])[0]


def _normal(J):
    """Phi^-1((J + 1/2) / 2^32) from the nearer tail."""
    up = J >= (1 << 31)
    z = torch.special.ndtri((torch.where(up, J ^ 0xFFFFFFFF, J).double() + 0.5) * 2.0 ** -32)
    return torch.where(up, -z, z)


class _Path:
    """Running state of one path and its payoff (fine, or coarse on its own grid)."""

    def __init__(self, S0, n):
        self.S, self.n = torch.full((n,), S0, dtype=torch.float64, device="cuda"), 0
        self.acc, self.low = 0.5 * self.S, self.S.clone()

    def step(self, inc):
        if self.n:
            self.acc = self.acc + self.S
        self.S = self.S + self.S * inc
        self.low = torch.minimum(self.low, self.S)
        self.n += 1

    def payoff(self, p):
        if p["payoff"] == W.DIGITAL:
            return (self.S > p["K"]).double()
        if p["payoff"] == W.LOOKBACK:
            return self.S - self.low
        x = (self.acc + 0.5 * self.S) / self.n if p["payoff"] == W.ASIAN else self.S
        return (x - p["K"]).clamp(min=0.0)


def _increment(p, h, z, m2):
    inc = p["r"] * h * m2 + p["sigma"] * math.sqrt(h) * z
    return inc + 0.5 * p["sigma"] ** 2 * h * (z * z - m2) if p["scheme"] == W.MILSTEIN else inc


def _rd(x, k):
    return (x + (1 << (k - 1))) >> k if k > 0 else x << -k


class _Fixed:
    """Algorithm 1 in the default formats' fractional bits (no variable saturates at six standard deviations)."""

    def __init__(self, p, level, d):
        h = p["T"] / (1 << level)
        f = {k: min(24, max(10, b + level * (k != "Z"))) for k, b in
             dict(Z=12, con1=16, con2=14, mul1=12, sum1=12, mul2=12, S=14).items()}
        f["S"] = min(f["S"], 21)
        smax = max(p["S0"] * math.exp(abs(p["r"]) * p["T"] + 6 * p["sigma"] * math.sqrt(p["T"])), p["K"])
        eS = math.floor(math.log2(smax + 2.0 ** -(f["S"] + 1))) + 1
        f["S"] = f["S"] if eS + f["S"] <= 30 else max(10, 30 - eS)
        f["mul2"] = min(f["mul2"], f["S"])
        q = lambda x, b: math.floor(x * 2.0 ** b + 0.5)  # noqa: E731
        self.f, self.p, self.d = f, p, d
        self.con1 = [q(p["r"] * h, f["con1"]), q(p["r"] * (2 * h), f["con1"])]
        self.con2, self.con3 = q(p["sigma"] * math.sqrt(h), f["con2"]), q(0.5 * p["sigma"] ** 2 * h, f["con1"])
        self.S0, self.K = q(p["S0"], f["S"]), q(p["K"], f["S"])
        # the mean of Phi^-1 over each of the 2^d intervals, mirrored about 1/2
        a = torch.special.ndtri(torch.arange((1 << (d - 1)) + 1, dtype=torch.float64) / (1 << d))
        phi = torch.exp(-0.5 * a * a) / math.sqrt(2 * math.pi)
        half = torch.floor((phi[:-1] - phi[1:]) * 2.0 ** (d + f["Z"]) + 0.5).long()
        self.z = torch.cat([half, -half.flip(0)]).cuda()

    def path(self, n):
        S = torch.full((n,), self.S0, dtype=torch.int64, device="cuda")
        return dict(S=S, inner=torch.zeros_like(S), low=S.clone(), n=0)

    def step(self, st, z, coarse):
        f = self.f
        F1, F2 = max(f["con1"], f["mul1"]), max(f["S"], f["mul2"])
        mul = _rd(self.con2 * z, f["con2"] + f["Z"] - f["mul1"])
        if self.p["scheme"] == W.MILSTEIN:
            mul = mul + _rd(self.con3 * (z * z - ((1 + coarse) << 2 * f["Z"])), f["con1"] + 2 * f["Z"] - f["mul1"])
        sum1 = _rd((self.con1[coarse] << (F1 - f["con1"])) + (mul << (F1 - f["mul1"])), F1 - f["sum1"])
        mul2 = _rd(st["S"] * sum1, f["S"] + f["sum1"] - f["mul2"])
        if st["n"]:
            st["inner"] = st["inner"] + st["S"]
        st["S"] = _rd((st["S"] << (F2 - f["S"])) + (mul2 << (F2 - f["mul2"])), F2 - f["S"])
        st["low"], st["n"] = torch.minimum(st["low"], st["S"]), st["n"] + 1

    def payoff(self, st):
        pay, unit = self.p["payoff"], 2.0 ** -self.f["S"]
        if pay == W.DIGITAL:
            return (st["S"] > self.K).double()
        if pay == W.LOOKBACK:
            return (st["S"] - st["low"]).double() * unit
        if pay == W.ASIAN:
            tot = self.S0 + 2 * st["inner"] + st["S"]
            return (tot - 2 * st["n"] * self.K).clamp(min=0).double() * unit / (2 * st["n"])
        return (st["S"] - self.K).clamp(min=0).double() * unit


def _sums(p, variant, level, N, seed, request=0, d=10):
    """Discounted sums of Y and Y^2 of an exact or a fixed-point correction estimator."""
    h, total, total2 = p["T"] / (1 << level), 0.0, 0.0
    fx = _Fixed(p, level, d) if variant == "corr_fixed" else None
    for at in range(0, N, 1 << 22):
        s = torch.arange(at, min(N, at + (1 << 22)), dtype=torch.int64, device="cuda")
        fine, coarse = _Path(p["S0"], len(s)), _Path(p["S0"], len(s))
        af, ac = (fx.path(len(s)), fx.path(len(s))) if fx else (None, None)
        for i, J in enumerate(_uniforms(s, level, seed, request)):
            z = _normal(J)
            fine.step(_increment(p, h, z, 1))
            if fx:
                za = fx.z[J >> (32 - d)]
                fx.step(af, za, 0)
            if i & 1:
                coarse.step(_increment(p, h, z0 + z, 2))
                if fx:
                    fx.step(ac, za0 + za, 1)
            else:
                z0, za0 = z, za if fx else None
        y = fine.payoff(p)
        if level:
            y = y - coarse.payoff(p)
        if fx:
            y = y - fx.payoff(af) + (fx.payoff(ac) if level else 0.0)
        total += float(y.sum())
        total2 += float((y * y).sum())
    disc = math.exp(-p["r"] * p["T"])
    return disc * total, disc * disc * total2


def _sens(p, level, N, seed):
    """Second moments of d(P_f - P_c)/dx for every Algorithm-1 intermediate x, by the chain rule
    (S_n depends on S_k+1 through the factor S_n / S_k+1)."""
    n, h, disc = 1 << level, p["T"] / (1 << level), math.exp(-p["r"] * p["T"])
    c1, c2, mc = p["r"] * h, p["sigma"] * math.sqrt(h), (1 << level) // 2
    ni = n + mc + 1
    inst = torch.zeros(7, ni, dtype=torch.float64, device="cuda")
    top, tot = torch.zeros(7, dtype=torch.float64, device="cuda"), [0.0, 0.0]
    for at in range(0, N, max(1, (1 << 23) >> level)):
        s = torch.arange(at, min(N, at + max(1, (1 << 23) >> level)), dtype=torch.int64, device="cuda")
        z = torch.stack([_normal(J) for J in _uniforms(s, level, seed)])
        sides = [(z, c1, n)] + ([(z[0::2] + z[1::2], 2 * c1, mc)] if mc else [])
        bars, zbar, dp = [], torch.zeros_like(z), 0.0
        for k, (zz, con1, steps) in enumerate(sides):
            sum1 = con1 + c2 * zz
            S = p["S0"] * torch.cumprod(1 + sum1, 0)
            prev = torch.cat([torch.full_like(S[:1], p["S0"]), S[:-1]])
            for t, x in ((0, z), (3, c2 * zz), (4, sum1), (5, prev * sum1), (6, S)):
                top[t] = torch.maximum(top[t], x.abs().max())
            sign = (1.0 - 2.0 * k) * disc * (S[-1] > p["K"]).double()
            dp = dp + sign * (S[-1] - p["K"])
            bS, b1 = sign * S[-1] / S, sign * S[-1] / (1 + sum1)
            zbar += c2 * (b1 if k == 0 else b1.repeat_interleave(2, 0))
            lo = k * n
            for t, b in ((3, b1), (4, b1), (5, bS), (6, bS)):
                inst[t, lo:lo + steps] += (b * b).sum(1)
            bars.append((sign * S[-1] / p["S0"], b1.sum(0), (b1 * zz).sum(0)))
            inst[1, k] += (bars[k][1] ** 2).sum()
        inst[0, :n] += (zbar * zbar).sum(1)
        inst[2, 0] += (sum(b[2] for b in bars) ** 2).sum()
        inst[6, n + mc] += (sum(b[0] for b in bars) ** 2).sum()
        tot = [tot[0] + float(dp.sum()), tot[1] + float((dp * dp).sum())]
    inst /= N
    top[6] = max(float(top[6]), p["S0"])
    top[1], top[2] = abs(c1) * (2 if mc else 1), abs(c2)
    mean = tot[0] / N
    return dict(A=inst.sum(1).tolist(), B=inst.sqrt().sum(1).tolist(), maxabs=top.tolist(), mean=mean,
                var=max(0.0, tot[1] / N - mean * mean), n=None, inst=inst.cpu().numpy())


def exact(case, seed):
    kind = case["kind"]
    if kind == "level" and case["variant"] in ("fp64", "fp32", "corr_fixed"):
        if case["variant"] == "corr_fixed" and case["method"] != 1:
            return None
        p, key = _of_level(case, seed)
        s, s2 = _sums(p, case["variant"], case["level"], case["N"], key, d=case["d"])
        return dict(sum=s, sum2=s2)
    if kind in ("list", "plan") and case["work"] != "nested":
        items, key = _items(case, seed)
        got = [_sums(p, v, lev, n, key, req) for p, v, lev, n, req, _ in items]
        return dict(sum=np.array([a for a, _ in got]), sum2=np.array([b for _, b in got]))
    if kind == "sens":
        p, key = _market(seed)
        return _sens(p, case["level"], case["N"], key)
    # sums of integers (compared bit for bit), 16-bit roundings, and schedules that follow the sums
    return None
