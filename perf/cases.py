"""Measured cases: what a program has this library do, through its public
entry points.

A case names one call: the level sums of a range of pairs (`run_level`, with
or without a context), one adaptive estimate (`estimate`), or a batch of
estimates (`estimate_batch`), on the problems of `workloads.py`: free space
from the origin, the periodic cosine density, and the paper's backgrounds
B1/B2.  The random numbers of a pass are the Philox streams of the seed.

`exact` restates the method in plain torch FP64 (Alg. 1, Alg. 2, the mapping
and aggregation of Sec. 3, the sample counts of Sec. 4.1), vectorised over
pairs, without this repository's code.
"""
import math

import numpy as np
import torch

import paper_2004_04071_gb300 as mk

PREC = {"fp64": mk.PREC_FP64, "fp64_u24": mk.PREC_FP64_U24, "fp32_dy64": mk.PREC_FP32_DY64,
        "fp32_comp": mk.PREC_FP32_COMP}
HETERO = {"b1": mk.BG_B1, "b2": mk.BG_B2}
SUMS = ("sy", "sy2", "sqf", "sqf2", "sqc", "sqc2")


def listed():
    return [
        # the smallest call of a session: the two-level free-space problem in the default precision
        dict(name="two_level_fp64", kind="level", shape="free", prec="fp64", eps=0.5, M=2, L=1, level=1, n=2000,
             first=0, nbins=20),
        # a warm-up round of 100 pairs from a host program that may not allocate on the device
        dict(name="noalloc_warmup_fp32", kind="noalloc", shape="periodic", prec="fp32_dy64", eps=0.1, M=2, L=8,
             level=5, n=100, first=0, nbins=0),
        # a finest coupled level in the default precision, kinetic to mixed regime, with the density
        dict(name="level8_fp64", kind="level", shape="periodic", prec="fp64", eps=0.1, M=2, L=8, level=8, n=131071,
             first=100, nbins=128),
        # the paths of the coarsest level, most of an estimate's samples: two events each
        dict(name="level0_fp64", kind="level", shape="periodic", prec="fp64", eps=0.1, M=2, L=8, level=0, n=500009,
             first=100, nbins=128),
        # a deep diffusive level: few pairs of thousands of serial events
        dict(name="deep_fp64", kind="level", shape="periodic", prec="fp64", eps=1e-3, M=2, L=12, level=10, n=1000,
             first=0, nbins=0),
        # the same finest coupled level in FP32, a throughput-bound launch
        dict(name="level8_fp32", kind="level", shape="periodic", prec="fp32_comp", eps=0.1, M=2, L=8, level=8,
             n=1000003, first=0, nbins=128),
        # the coarsest level of a density request in FP32
        dict(name="level0_fp32", kind="level", shape="density", prec="fp32_dy64", eps=0.1, M=2, L=8, level=0,
             n=4000037, first=0, nbins=64),
        # a fine level of the paper's symmetric heterogeneous background
        dict(name="hetero_b1_fp32", kind="level", shape="b1", prec="fp32_comp", a=10.0, b=1000.0, M=2, L=12,
             level=10, n=100003, first=0, nbins=0),
        # one adaptive estimate of E[x^2] in the default precision: warm-up, rounds, controller
        dict(name="estimate_fp64", kind="estimate", shape="free", prec="fp64", eps=0.3, M=2, L=4, tol=2e-3, nbins=0),
        # the periodic full-MLMC step at fixed counts, three estimates in one graph launch
        dict(name="batch_step_fp32", kind="batch", shape="periodic", prec="fp32_comp", eps_hi=1.0, eps_lo=1e-3,
             requests=3, M=2, cap=12, tol=1e-3, fixed=True, nbins=128, substeps=0, warp_pair=-1),
        # time to tolerance: the same three estimates from scratch, deep pairs one per warp
        dict(name="batch_adaptive_fp32", kind="batch", shape="periodic", prec="fp32_comp", eps_hi=1.0, eps_lo=1e-3,
             requests=3, M=2, cap=12, tol=1e-3, fixed=False, nbins=128, substeps=0, warp_pair=0),
        # a queue of small mixed requests in the default precision and the default slices
        dict(name="batch_requests_fp64", kind="batch", shape="mixed", prec="fp64", eps_hi=1.0, eps_lo=0.1,
             requests=8, M=2, cap=7, tol=2e-2, fixed=False, nbins=0, substeps=256, warp_pair=0),
    ]


#: KD events of a drawn case at most: a pass then takes no longer than the largest listed one.
MOST = {"fp64": 2.0e7, "fp64_u24": 2.0e7, "fp32_dy64": 6e8, "fp32_comp": 6e8}


def draw(rng):
    kind = rng.choice(["level"] * 6 + ["noalloc", "estimate", "estimate", "batch", "batch", "batch"])
    prec = rng.choice(["fp64", "fp64", "fp64_u24", "fp32_dy64", "fp32_comp", "fp32_comp"])
    fp64 = prec.startswith("fp64")
    log = lambda lo, hi: math.exp(rng.uniform(math.log(lo), math.log(hi)))  # noqa: E731
    while True:
        M = rng.choice([2, 2, 2, 3, 4, 8])
        if kind in ("level", "noalloc"):
            shape = rng.choice(["free", "periodic", "periodic", "density", "b1", "b2"])
            c = dict(kind=kind, shape=shape, prec=prec, M=M, nbins={"density": rng.choice([33, 64, 128])}.get(
                shape, 0 if shape in HETERO else rng.choice([0, 0, 20, 128])), first=rng.randrange(0, 10**6))
            if shape in HETERO:
                c.update(a=round(log(0.1, 100.0), 3), b=round(log(1.0, 1e4), 3))
            else:
                c["eps"] = round(log(1e-3, 1.0), 6)
            c["level"] = rng.randrange(0, 1 + int(math.log(1024 if fp64 else 4096, M)))
            c["L"] = c["level"]
            c["n"] = int(log(100, 4e6))
        elif kind == "estimate":
            c = dict(kind=kind, shape=rng.choice(["free", "periodic", "density"]), prec=prec, M=M,
                     eps=round(log(0.03, 1.0), 5), L=rng.randrange(1, 5), tol=round(log(1e-3, 2e-2), 6))
            c["nbins"] = 16 if c["shape"] == "density" else 0
            if c["shape"] == "density":
                c["tol"] = round(log(1e-2, 5e-2), 6)
        else:
            c = dict(kind=kind, shape=rng.choice(["free", "periodic", "mixed"]), prec=prec, M=2,
                     eps_hi=round(log(0.2, 1.0), 5), eps_lo=round(log(0.05 if fp64 else 3e-3, 0.2), 6),
                     requests=rng.randrange(1, 17), cap=8 if fp64 else 12, fixed=rng.random() < 0.3,
                     tol=round(log(1e-3, 2e-2), 6), nbins=rng.choice([0, 0, 64]), substeps=rng.choice([0, 0, 256]),
                     warp_pair=rng.choice([0, 0, -1, 4096]))
        work_ = [_request(c, j) for j in range(c.get("requests", 1))]
        events = sum(n * sum(_events(r, j)) for r in work_ for j, n in _counts(c, r))
        # batches of small FP64 requests spend more of a pass waiting for their longest chains
        if events <= MOST[prec] / (2 if c["shape"] in HETERO else 8 if kind == "batch" and fp64 else 1):
            return c


# ---------------------------------------------------------------------------
# Problems of a case
# ---------------------------------------------------------------------------
def _request(c, j=0):
    """Request j of a case: the arguments of make_problem, without seed and counts."""
    shape = c["shape"]
    if shape == "mixed":
        shape = "free" if j % 2 == 0 else "periodic"
    r = dict(M=c["M"], nbins=c["nbins"], n_warmup=100, request=j, precision=PREC[c["prec"]], tol=c.get("tol", 0.0))
    if shape in HETERO:
        r.update(eps=1.0, T=1.0, dt0=1.0, qoi=mk.QOI_X, init=mk.INIT_POINT, x0=1.0, background=HETERO[shape],
                 bg_a=c["a"], bg_b=c["b"])
    elif shape == "free":
        r.update(T=0.5, dt0=0.1, qoi=mk.QOI_X2, init=mk.INIT_ORIGIN, lo=-3.0, hi=3.0)
    else:
        r.update(T=1.0, dt0=0.5, qoi=mk.QOI_DENSITY if shape == "density" else mk.QOI_X2_PERIODIC,
                 init=mk.INIT_COSINE, lo=0.0, hi=1.0)
    if c["kind"] == "batch":
        f = j / (c["requests"] - 1) if c["requests"] > 1 else 0.0
        r["eps"] = c["eps_hi"] ** (1 - f) * c["eps_lo"] ** f
        if c["requests"] == 3:     # 1, 0.1, 1e-3: the periodic benchmark's three regimes
            r["eps"] = (c["eps_hi"], math.sqrt(c["eps_hi"] * c["eps_lo"] * 10), c["eps_lo"])[j]
        r["L"] = min(c["cap"], max(1, math.ceil(math.log2(r["dt0"] / (r["eps"] ** 2 / 4.0)))))
    else:
        r["L"] = c["L"]
        if "eps" in c:
            r["eps"] = c["eps"]
    return r


def _rate(r):
    return r["bg_b"] if "background" in r else 1.0 / r["eps"] ** 2


def _steps(r, level):
    return int(round(r["T"] / r["dt0"])) * r["M"] ** level


def _events(r, level):
    """Expected (fine, coarse) KD events of a pair: each step holds a collision
    with probability 1 - exp(-R dt), on both paths."""
    n, z = _steps(r, level), _rate(r) * r["dt0"] / r["M"] ** level
    return -n * math.expm1(-z), -n / r["M"] * math.expm1(-z * r["M"]) if level else 0.0


def _counts(c, r):
    """(level, pairs) of a case's request: given, or about the counts of eqs.
    Nopt1/Noptj, for level variances that fall like dt^3 below R dt = 1 and
    like dt^-3.6 above R dt = 50, as the periodic problem's do."""
    if "n" in c:
        return [(c["level"], c["n"])]
    v, cost = [], []
    for l in range(r["L"] + 1):
        z = _rate(r) * r["dt0"] / r["M"] ** l
        v0 = 0.09 if r["init"] == mk.INIT_COSINE else 2.0
        if r["qoi"] == mk.QOI_DENSITY:
            v0 = float(r["nbins"])
        v.append(v0 if l == 0 else 2.0 * v0 / (z ** -3.0 + 1.0 + (z / 50.0) ** 3.6))
        cost.append(sum(_events(r, l)))
    total = sum(math.sqrt(a * b) for a, b in zip(v, cost))
    return [(l, max(r["n_warmup"], math.ceil(2.0 / r["tol"] ** 2 * math.sqrt(v[l] / cost[l]) * total)))
            for l in range(r["L"] + 1)]


# ---------------------------------------------------------------------------
# What a program has in hand, one pass, and what the pass cannot do without
# ---------------------------------------------------------------------------
def prepare(case, seed):
    c = case
    problems = []
    for j in range(c.get("requests", 1)):
        r = _request(c, j)
        fixed = [n for _, n in _counts(c, r)] if c.get("fixed") else None
        problems.append(mk.make_problem(seed=seed, n_fixed=fixed, **r))
    state = dict(case=c, problems=problems)
    if c["kind"] == "batch":
        state["cfg"] = mk.batch_config(substeps_per_launch=c["substeps"], max_requests=max(16, c["requests"]),
                                       warp_pair_min_events=c["warp_pair"])
        state["ctx"] = mk.Context(0, arena_bytes=mk.batch_workspace_bytes(state["cfg"]))
    elif c["kind"] != "noalloc":
        state["ctx"] = mk.Context(0)
    return state


def _fields(results):
    """Every field of the results of one call, levels and requests one after another."""
    out = {k: np.array([lv[k] for r in results for lv in r.levels]) for k in ("n", "events_f", "events_c") + SUMS}
    out["estimate"] = np.array([r.estimate for r in results])
    out["variance"] = np.array([r.variance for r in results])
    out["rounds"] = np.array([r.rounds for r in results])
    out["var_level"] = np.array([v for r in results for v in r.var_level])
    out["cost_level"] = np.array([v for r in results for v in r.cost_level])
    if results[0].density is not None:
        out["density"] = np.concatenate([r.density for r in results])
    return out


def run(state):
    c, problems = state["case"], state["problems"]
    if c["kind"] == "level":
        return state["ctx"].run_level(problems[0], c["level"], c["first"], c["n"])
    if c["kind"] == "noalloc":
        return mk.run_level_noalloc(problems[0], c["level"], c["first"], c["n"])
    if c["kind"] == "estimate":
        return _fields([state["ctx"].estimate(problems[0])])
    return _fields(state["ctx"].estimate_batch(problems, state["cfg"]))


def work(case):
    """Bytes: the results.  Operations: about 190 per fine and 50 per coarse
    event (random numbers, transforms, coefficients, weights, updates), and
    about 300 per pair (its draw, initial position and summation)."""
    flops, nbytes = 0.0, 0.0
    for j in range(case.get("requests", 1)):
        r = _request(case, j)
        for level, n in _counts(case, r):
            f, k = _events(r, level)
            flops += n * (190.0 * f + 50.0 * k + 300.0)
            nbytes += 72.0 + 24.0 * r["nbins"]
    return {"bytes": nbytes, "flops": flops}


# ---------------------------------------------------------------------------
# The method in plain torch FP64
# ---------------------------------------------------------------------------
def _philox(c, seed):
    """Philox4x32-10 (SC'11) on int64 tensors holding 32-bit words."""
    low = 0xFFFFFFFF
    k0, k1 = seed & low, (seed >> 32) & low
    for _ in range(10):
        pa, pb = c[0] * 0xD2511F53, c[2] * 0xCD9E8D57
        c = [((pb >> 32) & low) ^ c[1] ^ k0, pb & low, ((pa >> 32) & low) ^ c[3] ^ k1, pa & low]
        k0, k1 = (k0 + 0x9E3779B9) & low, (k1 + 0xBB67AE85) & low
    return c


def _draw(P, k, pair):
    """nu, chi, E and the fourth uniform of block k of these pairs."""
    def block(tag):
        full = lambda v: torch.full_like(pair, v)  # noqa: E731
        return _philox([full(k), pair & 0xFFFFFFFF, (pair >> 32) ^ (P["level"] << 24) ^ (tag << 16),
                        full(P["request"])], P["seed"])
    a = block(0)
    if P["u24"]:
        u = [((w >> 8) + 1).double() * 2.0**-24 for w in a]
    else:
        b = block(1)
        u = [(((x << 21) ^ (y >> 11)) + 1).double() * 2.0**-53 for x, y in ((a[0], a[1]), (a[2], a[3]), (b[0], b[1]),
                                                                            (b[2], b[3]))]
    rad = torch.sqrt(-2.0 * torch.log(u[0]))
    return rad * torch.cos(2 * math.pi * u[1]), rad * torch.sin(2 * math.pi * u[1]), -torch.log(u[2]), u[3]


def _series(s, lead, term):
    """sum_{n >= lead} (-1)^n term(n) s^n / n! for 0 <= s < 1."""
    p = torch.zeros_like(s)
    for n in range(26, lead - 1, -1):
        p = p * s + (-1) ** n * term(n) / math.factorial(n)
    return p * s**lead


def _h(s):
    return torch.where(s < 1, _series(s.clamp(max=1), 2, lambda n: 1), torch.exp(-s) + s - 1)


def _kd(R, sigma, theta, dv):
    """eqs. advection and diffusion (mu = 0), h(s) and 1 - exp(-s) at s = R theta."""
    s = R * theta
    t, e, small = s.clamp(max=1), torch.exp(-s), s < 1
    f = torch.where(small, _series(t, 3, lambda n: 2 - n), 2 * (e - 1) + s * (e + 1))
    g = torch.where(small, _series(t, 3, lambda n: 2 * n - 2**n), 1 - 2 * s * e - e * e)
    h = _h(s)
    om = s - h
    d = torch.sqrt((2 * (sigma / R) ** 2 * f + (dv / R) ** 2 * g).clamp(min=0))
    return dv * om / R, d, h, om


def _start(P, u):
    """Initial positions: a point, or the inverse CDF of 1 + cos(2 pi x)."""
    if not P["cosine"]:
        return torch.full_like(u, P["x0"])
    lo, hi = torch.full_like(u, -0.5), torch.full_like(u, 0.5)
    for _ in range(60):
        y = 0.5 * (lo + hi)
        z = 2 * math.pi * y
        small = sum((-1) ** (i + 1) * z ** (2 * i + 1) / float(math.factorial(2 * i + 1)) for i in range(1, 12))
        G = torch.where(z.abs() < 1, small, z - torch.sin(z)) / (2 * math.pi)
        below = G < u - 0.5
        lo, hi = torch.where(below, y, lo), torch.where(below, hi, y)
    x = 0.5 * (lo + hi) + 0.5
    return torch.where(x >= 1, x - 1, x)


def _slopes(P, x, v):
    """Rate at x, and its change per step along v before and after x = 1 (in steps)."""
    right, left = torch.full_like(x, P["b"] * P["a_right"]), torch.full_like(x, -P["b"] * P["a_left"])
    rate = P["b"] * (1 + P["a_left"] * (1 - x).clamp(min=0) + P["a_right"] * (x - 1).clamp(min=0))
    side = lambda y: torch.where((y > 1) | ((y == 1) & (v > 0)), right, left)  # noqa: E731
    s1, s2 = side(x) * v * P["dt"] ** 2, side(torch.ones_like(x)) * v * P["dt"] ** 2
    kink = torch.where((s1 == s2) | (v == 0) | (x == 1), -torch.ones_like(x), (1 - x) / (v * P["dt"]))
    return rate * P["dt"], s1, s2, kink


def _depth(P, x, v, u):
    """Integral of R over u steps of the path from x (negative behind it)."""
    back = u < 0
    x, w = torch.where(back, x + v * P["dt"] * u, x), u.abs()
    rho, s1, s2, kink = _slopes(P, x, v)
    past = (kink > 0) & (w > kink)
    a = torch.where(past, kink, w)
    r = w - a
    total = rho * a + 0.5 * s1 * a * a + torch.where(past, P["b"] * P["dt"] * r + 0.5 * s2 * r * r, torch.zeros_like(r))
    return torch.where(back, -total, total)


def _flight(P, x, v, E):
    """Steps until the integral of R along the path reaches E (eq. intinv)."""
    rho, s1, s2, kink = _slopes(P, x, v)
    root = lambda p, s, e: 2 * e / (p + torch.sqrt((p * p + 2 * s * e).clamp(min=0)))  # noqa: E731
    first = rho * kink + 0.5 * s1 * kink * kink
    past = (kink > 0) & (E > first)
    second = kink + root(P["b"] * P["dt"], s2, torch.where(past, E - first, E))
    return torch.where(past, second, root(rho, s1, E))


def _pairs(P, first, count, device):
    """Positions at T and KD events of pairs [first, first + count): Alg. 1 and
    Alg. 2 in steps of the fine grid, all pairs one event at a time."""
    n, M, dt, coupled, het = P["n"], P["M"], P["dt"], P["coupled"], P["het"]
    pair = torch.arange(first, first + count, dtype=torch.int64, device=device)
    out = [torch.zeros(count, dtype=torch.float64, device=device) for _ in range(4)]
    nu, _, E, u = _draw(P, 0, pair)
    x = _start(P, u)
    v = P["sigma"] * nu
    top = 4 * n + 4
    q = _flight(P, x, v, E) if het else E / (P["R"] * dt)
    zero, one = torch.zeros_like(x), torch.ones_like(x)
    # fine x v q i; coarse x v q i; window num den first fresh; events; kept output x v i, kept; pair; place
    S = dict(xf=x, vf=v, qf=q, jf=zero, xc=x.clone(), vc=v.clone(), qc=q.clone(), jc=zero, num=zero, den=zero,
             chi=zero, fresh=one, ef=zero, ec=zero, xo=x, vo=v, jo=zero, kept=zero, pair=pair,
             at=torch.arange(count, device=device))
    k = 0
    while True:
        fine_left = S["qf"] < n - S["jf"]
        coarse_left = (S["qc"] < n - S["jc"]) if coupled else torch.zeros_like(fine_left)
        keep = (S["kept"] == 0) & ~fine_left      # the fine state at its first collision past T
        for o, s in (("xo", "xf"), ("vo", "vf"), ("jo", "jf")):
            S[o] = torch.where(keep, S[s], S[o])
        S["kept"] = torch.where(keep, one[: len(keep)], S["kept"])
        live = fine_left | coarse_left
        end = ~live
        if bool(end.any()):
            F = {a: b[end] for a, b in S.items()}
            at = F["at"]
            drift = lambda x, v, j: x + v * ((n - j).clamp(min=0) * dt)  # noqa: E731
            out[0][at] = drift(F["xo"], F["vo"], F["jo"])
            if coupled:
                out[1][at] = drift(F["xc"], F["vc"], F["jc"])
            out[2][at], out[3][at] = F["ef"], F["ec"]
            S = {a: b[live] for a, b in S.items()}
            if len(S["at"]) == 0:
                return out
        k += 1
        nu, chi, E, _ = _draw(P, k, S["pair"])
        sq = torch.floor(S["qf"].clamp(max=top))
        theta = dt * (sq + 1 - S["qf"]).clamp(min=0) if het else dt * (sq + 1 - S["qf"])
        hit = S["xf"] + S["vf"] * (S["qf"] * dt)
        R = _slopes(P, hit, S["vf"])[0] / dt if het else torch.full_like(hit, P["R"])
        dv = P["sigma"] * nu
        a, d, h, om = _kd(R, P["sigma"], theta, dv)
        bound = M * (torch.floor((S["jc"] + torch.floor(S["qc"].clamp(max=top))) / M) + 1)
        S["xf"], S["vf"] = hit + a + d * chi, dv
        S["jf"] = (S["jf"] + sq + 1).clamp(max=top)
        S["qf"] = _flight(P, S["xf"], dv, E) if het else E / (P["R"] * dt)
        S["ef"] = S["ef"] + 1
        if not coupled:
            continue
        beta = torch.sqrt(2 * _h(h)) * P["sigma"] / R
        S["chi"] = torch.where(S["fresh"] > 0, chi, S["chi"])
        S["num"], S["den"] = S["num"] + beta * chi, S["den"] + beta * beta
        closes = S["jf"] + torch.floor(S["qf"].clamp(max=top)) >= bound
        alpha = P["sigma"] * (S["qf"] * dt + om / R)
        chit = torch.where(S["den"] > 0, S["num"] / torch.sqrt(S["den"].clamp(min=1e-300)), S["chi"])
        thc = dt * (bound - S["jc"] - S["qc"])
        hitc = S["xc"] + S["vc"] * (S["qc"] * dt)
        Rc = _slopes(P, hitc, S["vc"])[0] / dt if het else R
        ac, dc, _, _ = _kd(Rc, P["sigma"], thc.clamp(min=0), dv)
        xc = hitc + ac + dc * chit
        if het:
            qc = _flight(P, xc, dv, E - _depth(P, S["xf"], dv, bound - S["jf"]))
        else:
            qc = S["qf"] - (bound - S["jf"])
        go = closes & (S["qc"] < n - S["jc"])     # the coarse KD step, while the coarse path is before T
        for name, new in (("xc", xc), ("vc", dv), ("qc", qc), ("jc", bound.clamp(max=top)), ("ec", S["ec"] + 1)):
            S[name] = torch.where(go, new, S[name])
        none = torch.zeros_like(xc)
        S["num"] = torch.where(closes, none, S["num"] + alpha * nu)
        S["den"] = torch.where(closes, none, S["den"] + alpha * alpha)
        S["fresh"] = closes.double()


def _level_sums(r, seed, level, first, count, device):
    het = "background" in r
    P = dict(n=_steps(r, level), M=r["M"], dt=r["dt0"] / r["M"] ** level, coupled=level > 0, het=het, R=_rate(r),
             sigma=1.0 if het else 1.0 / r["eps"], level=level, request=r["request"], seed=seed,
             u24=r["precision"] != mk.PREC_FP64, cosine=r["init"] == mk.INIT_COSINE, x0=r.get("x0", 0.0))
    if het:
        P.update(b=r["bg_b"], a_left=r["bg_a"] if r["background"] == mk.BG_B1 else 0.0, a_right=r["bg_a"])
    periodic = r["init"] == mk.INIT_COSINE
    total, hist = dict.fromkeys(SUMS + ("events_f", "events_c"), 0.0), np.zeros((3, r["nbins"]))
    for lo in range(first, first + count, 1 << 20):
        xf, xc, ef, ec = _pairs(P, lo, min(1 << 20, first + count - lo), device)
        wrap = (lambda x: x - torch.floor(x)) if periodic else (lambda x: x)
        F = (lambda x: x) if r["qoi"] == mk.QOI_X else (lambda x: wrap(x) ** 2)
        qf, qc = F(xf), F(xc) if level else torch.zeros_like(xf)
        y = qf - qc if periodic or het else (xf - xc) * (xf + xc) if level else qf
        for name, t in zip(SUMS + ("events_f", "events_c"), (y, y * y, qf, qf * qf, qc, qc * qc, ef, ec)):
            total[name] += float(t.sum())
        if r["nbins"]:
            nb, a, b = r["nbins"], r["lo"], r["hi"]
            place = lambda x: torch.where((x >= a) & (x < b), ((x - a) / ((b - a) / nb)).floor().clamp(max=nb - 1),  # noqa: E731
                                          -torch.ones_like(x))
            bf, bc = place(wrap(xf)), place(wrap(xc)) if level else -torch.ones_like(xf)
            for row, t in enumerate((bf[bf >= 0], bc[bc >= 0], bf[(bf == bc) & (bf >= 0)])):
                hist[row] += torch.bincount(t.long(), minlength=nb).cpu().numpy()
    total["hist"] = hist
    return total


def _estimate(r, seed, counts, device):
    """One estimate: the given counts, or warm-up and rounds of Sec. 4.1."""
    nl = r["L"] + 1
    have, sums = [0] * nl, [None] * nl
    want = counts or [r["n_warmup"]] * nl
    h = (r["hi"] - r["lo"]) / r["nbins"] if r["nbins"] else 1.0
    spent = 0.0
    for rounds in range(65):
        spent += sum(max(0, want[l] - have[l]) * sum(_events(r, l)) for l in range(nl))
        if spent > MOST["fp64"] * 10:
            return None, spent
        for l in range(nl):
            if want[l] > have[l]:
                s = _level_sums(r, seed, l, have[l], want[l] - have[l], device)
                sums[l] = s if sums[l] is None else {k: sums[l][k] + s[k] for k in s}
                have[l] = want[l]
        var, cost = [], []
        for l in range(nl):
            s, m = sums[l], have[l]
            if r["qoi"] == mk.QOI_DENSITY:
                d, d2 = s["hist"][0] - s["hist"][1], s["hist"][0] + s["hist"][1] - 2 * s["hist"][2]
                v = ((d2 - d * d / m) / (m - 1)).max() / h**2
            else:
                v = (s["sy2"] - s["sy"] ** 2 / m) / (m - 1)
            var.append(max(0.0, float(v)))
            cost.append((s["events_f"] + s["events_c"]) / m)
        total = sum(math.sqrt(v * c) for v, c in zip(var, cost))
        want = [math.ceil(2.0 / r["tol"] ** 2 * math.sqrt(v / c) * total) if v > 0 and c > 0 else 0
                for v, c in zip(var, cost)]
        if counts or all(w <= m for w, m in zip(want, have)):
            break
    out = {k: [s[k] for s in sums] for k in SUMS}
    out.update(estimate=[sum(s["sy"] / m for s, m in zip(sums, have))], variance=[sum(v / m for v, m in zip(var, have))],
               var_level=var, cost_level=cost)
    if r["nbins"]:
        out["density"] = list(sum((s["hist"][0] - s["hist"][1]) / m for s, m in zip(sums, have)) / h)
    return out, spent


def exact(case, seed):
    device = "cuda" if torch.cuda.is_available() else "cpu"
    c = case
    requests = [_request(c, j) for j in range(c.get("requests", 1))]
    if sum(n * (sum(_events(r, l)) + 1) for r in requests for l, n in _counts(c, r)) > MOST["fp64"] * 10:
        return None
    if sum(_events(r, l)[0] for r in requests for l, _ in _counts(c, r)) * (1 if "n" in c or c.get("fixed") else 4) > 5000:
        return None     # events one after another
    if c["kind"] in ("level", "noalloc"):
        s = _level_sums(requests[0], seed, c["level"], c["first"], c["n"], device)
        # in B1 E[Y] = 0 by symmetry: in FP32 the sum of Y over few pairs is rounding
        noise = c["shape"] == "b1" and c["prec"].startswith("fp32")
        return {k: None if k == "sy" and noise else s[k] for k in SUMS}
    spent, parts = 0.0, []
    for r in requests:
        e, more = _estimate(r, seed, [n for _, n in _counts(c, r)] if c.get("fixed") else None, device)
        spent += more
        if e is None or spent > MOST["fp64"] * 10:
            return None
        parts.append(e)
    return {k: np.array([v for e in parts for v in e[k]]) for k in parts[0]}
