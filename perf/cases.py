"""The calls whose speed is tracked: what a program that uses this library has it do.

Every case runs through the public binding (`paper_2511_01573_gb300.gmq`, `autograd`).  The integrands are
the seeded Genz families with the difficulties of `genz_inputs`; sizes are those of the library's own
workloads (d = 3 product peak, d = 8 families, d = 12 mixed, uneven batches, d = 6 Gaussian gradients) and
ragged sizes in between.
"""
import itertools
import math
from decimal import Decimal, localcontext

import numpy as np
import torch

from paper_2511_01573_gb300 import autograd, gmq
from paper_2511_01573_gb300 import genz_inputs as G

FAMILIES = {"oscillatory": G.OSCILLATORY, "product_peak": G.PRODUCT_PEAK, "corner_peak": G.CORNER_PEAK,
            "gaussian": G.GAUSSIAN, "c0": G.C0, "discontinuous": G.DISCONTINUOUS}

# nominal arithmetic of one node: the inner sum's last step, the outer function, the accumulation
NODE_FLOPS = {"oscillatory": 22, "product_peak": 9, "corner_peak": 15, "gaussian": 15, "c0": 15, "discontinuous": 15}


def listed():
    return [
        # the smallest whole integration: one sweep of 4096 regions, launches and latency count
        {"name": "integrate_d3_peak", "kind": "integrate", "family": "product_peak", "dim": 3, "tol": 1e-6,
         "cap": 100000, "mixed": False},
        # a refining smooth integration: sweeps of all lengths up to some ten thousand regions
        {"name": "integrate_d8_corner", "kind": "integrate", "family": "corner_peak", "dim": 8, "tol": 1e-5,
         "cap": 1 << 22, "mixed": False},
        # a whole integration that refines to millions of regions (integrand with kinks)
        {"name": "integrate_d8_c0", "kind": "integrate", "family": "c0", "dim": 8, "tol": 1e-6,
         "cap": 1 << 22, "mixed": False},
        # the mixed-precision form of a refining integration
        {"name": "integrate_d8_c0_mixed", "kind": "integrate", "family": "c0", "dim": 8, "tol": 1e-5,
         "cap": 1 << 22, "mixed": True},
        # one large sweep's rule evaluation in FP64, the step a user's own loop calls
        {"name": "rule_d8_osc", "kind": "rule", "family": "oscillatory", "dim": 8, "n": 262144, "mixed": False,
         "null": False},
        # the same in a low dimension with a long ragged list
        {"name": "rule_d5_c0", "kind": "rule", "family": "c0", "dim": 5, "n": 1000003, "mixed": False,
         "null": False},
        # high dimension (4409 nodes a region), the null-rule error estimate
        {"name": "rule_d12_gauss", "kind": "rule", "family": "gaussian", "dim": 12, "n": 30011, "mixed": False,
         "null": True},
        # high dimension in mixed precision
        {"name": "rule_d12_corner_mixed", "kind": "rule", "family": "corner_peak", "dim": 12, "n": 200001,
         "mixed": True, "null": False},
        # many independent integrals of uneven dimension and tolerance in one device loop
        {"name": "batch_96", "kind": "batch", "count": 96, "tol": 1e-6},
        # value and gradient of a parametric integral, forward and backward through autograd
        {"name": "autograd_d6_gauss", "kind": "autograd", "dim": 6, "rows": 4, "tol": 1e-7},
        # the tensor Gauss-Kronrod rule (50625 nodes a region)
        {"name": "gk_d4_c0", "kind": "gk", "family": "c0", "dim": 4, "n": 2500},
        # one sweep's classification and bisection, half of a ragged list split
        {"name": "classify_split_d8", "kind": "classify", "dim": 8, "n": 3000017},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["integrate", "integrate", "rule", "rule", "mixed_rule", "mixed_integrate", "batch", "autograd",
                       "gk", "classify"])
    if kind in ("integrate", "mixed_integrate"):
        # dimensions and tolerances at which a family is refined, or stops with an estimate well above rounding
        family, low, high, tol = rng.choice([("oscillatory", 7, 8, -5.0), ("gaussian", 8, 8, -6.0),
                                             ("corner_peak", 7, 8, -5.0), ("c0", 3, 8, -6.0),
                                             ("product_peak", 3, 4, -6.0), ("discontinuous", 2, 4, -4.0)])
        mixed = kind == "mixed_integrate"
        return {"kind": "integrate", "family": family, "dim": rng.randint(low + (mixed and low == 2), high),
                "tol": 10.0 ** rng.uniform(max(tol, -5.0) if mixed else tol, -3.0), "cap": 1 << rng.randint(19, 22),
                "mixed": mixed}
    if kind in ("rule", "mixed_rule"):
        mixed = kind == "mixed_rule"
        family = rng.choice(list(FAMILIES))
        d = rng.randint(5 if family == "corner_peak" else 3 if mixed else 2, 12)
        most = int((8e8 if mixed else 1.3e8) / _nodes(d))
        return {"kind": "rule", "family": family, "dim": d, "n": _log_int(rng, 37, min(2000000, most)),
                "mixed": mixed, "null": rng.random() < 0.25}
    if kind == "batch":
        return {"kind": "batch", "count": rng.randint(8, 96), "tol": 10.0 ** rng.uniform(-6.0, -4.0)}
    if kind == "autograd":
        return {"kind": "autograd", "dim": rng.randint(2, 6), "rows": rng.randint(1, 4),
                "tol": 10.0 ** rng.uniform(-7.0, -4.0)}
    if kind == "gk":
        d = rng.randint(2, 5)
        return {"kind": "gk", "family": rng.choice(["c0", "product_peak"]), "dim": d,
                "n": _log_int(rng, 5, min(20000, int(1.3e8 / 15 ** d)))}
    return {"kind": "classify", "dim": rng.randint(2, 12), "n": _log_int(rng, 1000, 3000017)}


# ---- inputs ---------------------------------------------------------------

def _nodes(d):
    return (1 << d) + 2 * d * d + 2 * d + 1


def _params(case, seed):
    """Seeded parameters: the difficulties of the library's own workloads; the single sweeps of smooth families
    with the paper's f1 slopes and those of the gradient sets, whose error estimates are far above rounding."""
    family, d, f = case["family"], case["dim"], FAMILIES[case["family"]]
    if family == "product_peak":
        a, u = G.seed_uniform(seed, f, d, 4.5, 5.5)
        return a, 0.4 + 0.2 * u
    if family == "discontinuous":
        a, u = G.seed_genz(seed, f, d, 0.6 * d)
        return a, 0.3 + 0.6 * u
    if case["kind"] == "rule" and family in ("oscillatory", "gaussian"):
        return G.seed_uniform(seed, f, d, *((1.0, float(d)) if family == "oscillatory" else (0.5, 3.0)))
    return G.seed_genz(seed, f, d, G.GENZ_TARGET_SUM[f])


def _boxes(d, n, seed, coarse=False):
    """n sub-boxes of [0,1]^d as bisections leave them, up to some 24 / d in each axis: [d, n] centres and
    half-widths on the GPU.  `coarse`: the first sweeps of a rule of high degree, up to two in each axis."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    j = torch.randint(0, 3, (d, n), generator=g, device="cuda") if coarse else \
        torch.randint(1, 2 + 24 // d, (d, n), generator=g, device="cuda")
    h = torch.ldexp(torch.ones((), dtype=torch.float64, device="cuda"), -(j + 1))
    i = torch.floor(torch.rand((d, n), generator=g, device="cuda", dtype=torch.float64) * torch.ldexp(
        torch.ones((), dtype=torch.float64, device="cuda"), j))
    return (2.0 * i + 1.0) * h, h


def _batch_problems(case, seed):
    """Uneven dimensions and tolerances over the four families."""
    g = G.SplitMix64(seed)
    out = []
    for i in range(case["count"]):
        d = 2 + g.next_u64() % 7
        f = G.GENZ_D8_FAMILIES[g.next_u64() % 4]
        tol = case["tol"] * 10.0 ** (2.0 * g.next_double())
        a, u = G.seed_genz(seed * 8192 + i, f, int(d), G.GENZ_TARGET_SUM[f])
        out.append(G.Problem(f, int(d), a, u, tol))
    return out


def _grad_rows(case, seed):
    sets = [G.seed_uniform(seed * 65536 + i, G.GAUSSIAN, case["dim"], 0.5, 3.0) for i in range(case["rows"])]
    return np.stack([s[0] for s in sets]), np.stack([s[1] for s in sets])


def _classify_inputs(case, seed):
    """A sweep's rule outputs: errors spread over four decades around their share of the budget, half above."""
    d, n = case["dim"], case["n"]
    c, h = _boxes(d, n, seed)
    g = torch.Generator(device="cuda").manual_seed(seed + 1)
    vf = torch.prod(2.0 * h, dim=0)
    i7 = vf * (0.5 + torch.rand(n, generator=g, device="cuda", dtype=torch.float64))
    rank = torch.empty(n, device="cuda", dtype=torch.float64)
    rank[torch.randperm(n, generator=g, device="cuda")] = torch.arange(n, device="cuda", dtype=torch.float64)
    err = 1e-4 * vf * torch.exp(4.6 * (2.0 * (rank + 0.25) / n - 1.0))
    axis = torch.randint(0, d, (n,), generator=g, device="cuda").to(torch.uint8)
    return c, h, i7, err, vf, axis, 1e-4


def prepare(case, seed):
    ctx = gmq.Context(0)
    k = case["kind"]
    s = {"kind": k, "ctx": ctx}
    if k in ("integrate", "rule", "gk"):
        s["family"] = FAMILIES[case["family"]]
        s["a"], s["u"] = _params(case, seed)
    if k == "integrate":
        s["tol"], s["cap"] = case["tol"], case["cap"]
        s["precision"] = gmq.MIXED if case["mixed"] else gmq.FP64
    elif k in ("rule", "gk"):
        s["c"], s["h"] = _boxes(case["dim"], case["n"], seed, k == "gk")
        if k == "rule":
            s["precision"] = gmq.MIXED if case["mixed"] else gmq.FP64
            s["estimator"] = gmq.EST_NULL_RULES if case["null"] else gmq.EST_EMBEDDED
    elif k == "batch":
        s["problems"] = _batch_problems(case, seed)
    elif k == "autograd":
        a, u = _grad_rows(case, seed)
        s["a"], s["u"], s["tol"] = torch.tensor(a, device="cuda"), torch.tensor(u, device="cuda"), case["tol"]
    else:
        s["args"] = _classify_inputs(case, seed)
    return s


def _result(rs):
    return {"integral": np.array([r.integral for r in rs]), "error": np.array([r.error for r in rs]),
            "counts": np.array([(r.regions_evaluated, r.function_evals, r.final_active, r.iterations, r.status)
                                for r in rs], dtype=np.int64)}


def run(s):
    k, ctx = s["kind"], s["ctx"]
    if k == "integrate":
        return _result([ctx.integrate(s["family"], s["a"], s["u"], s["tol"], max_regions=s["cap"],
                                      precision=s["precision"])])
    if k == "rule":
        return list(ctx.eval_rule(s["family"], s["a"], s["u"], s["c"], s["h"], precision=s["precision"],
                                  estimator=s["estimator"]))
    if k == "gk":
        return list(ctx.eval_rule_gk(s["family"], s["a"], s["u"], s["c"], s["h"]))
    if k == "batch":
        return _result(ctx.integrate_batch(s["problems"], max_regions=1 << 20, pool_regions=1 << 23))
    if k == "autograd":
        a = s["a"].clone().requires_grad_(True)
        u = s["u"].clone().requires_grad_(True)
        v = autograd.integral(a, u, gmq.GAUSSIAN, s["tol"], ctx)
        v.sum().backward()
        return [v.detach(), a.grad, u.grad]
    c, h, i7, err, vf, axis, budget = s["args"]
    r = ctx.classify_split(c, h, i7, err, vf, axis, budget)
    return {"n_split": r["n_split"], "sums": np.array([r["ret_i"], r["ret_e"]]), "flags": r["flags"],
            "center": r["center"], "halfw": r["halfw"]}


def _nominal_regions(family, d, tol):
    """About how many regions an integration evaluates (the count depends on the drawn parameters)."""
    s = max(1, int(math.floor(4096 ** (1.0 / d) + 1e-9)))
    grow = {"oscillatory": 0.6, "gaussian": 0.1, "corner_peak": 1.2, "c0": 0.2 * d - 0.3, "product_peak": 0.4,
            "discontinuous": 1.2}[family] * (d / 8.0 if family == "corner_peak" else 1.0)
    return float(s ** d) * max(1.0, (1e-3 / tol) ** grow)


def work(case):
    k = case["kind"]
    if k == "integrate":
        d = case["dim"]
        n = _nominal_regions(case["family"], d, case["tol"])
        return {"bytes": n * 32 * d, "flops": n * _nodes(d) * NODE_FLOPS[case["family"]]}
    if k == "rule":
        d, n = case["dim"], case["n"]
        return {"bytes": n * (16 * d + 25), "flops": n * _nodes(d) * NODE_FLOPS[case["family"]]}
    if k == "gk":
        d, n = case["dim"], case["n"]
        return {"bytes": n * (16 * d + 25), "flops": float(n) * 15 ** d * (NODE_FLOPS[case["family"]] + 8)}
    if k == "batch":
        n = 5000.0 * case["count"] * (1e-4 / case["tol"]) ** 0.6
        return {"bytes": n * 32 * 5, "flops": n * _nodes(5) * 15}
    if k == "autograd":
        d = case["dim"]
        n = case["rows"] * 4096.0 * max(1.0, (1e-5 / case["tol"]) ** 0.6)
        return {"bytes": n * 48 * d, "flops": n * _nodes(d) * (2 * 15 + 4 * d)}
    # flag, axis and rule outputs of every region; centre and half-width of the half that is split, read once,
    # and of its two children, written once
    d, n = case["dim"], case["n"]
    return {"bytes": n * 27 + 0.5 * n * 48 * d, "flops": 4.0 * n}


# ---- the same results in 64 bits, without the library ----------------------

def _f64(family, a, u, x):
    """f at the nodes x [..., d]."""
    if family == "oscillatory":
        return torch.cos(2.0 * math.pi * u[0] + (x * a).sum(-1))
    if family == "product_peak":
        return 1.0 / torch.prod(a ** -2 + (x - u) ** 2, dim=-1)
    if family == "corner_peak":
        return (1.0 + (x * a).sum(-1)) ** -(x.shape[-1] + 1)
    if family == "gaussian":
        return torch.exp(-((a * (x - u)) ** 2).sum(-1))
    if family == "c0":
        return torch.exp(-(a * (x - u).abs()).sum(-1))
    return torch.where((x > u).any(-1), 0.0, torch.exp((x * a).sum(-1)))


def _gm_rule(d):
    """Node offsets in half-widths [N, d] and the degree-7 and degree-5 weights [N], unit volume."""
    l2, l3, l5 = math.sqrt(9 / 70), math.sqrt(9 / 10), math.sqrt(9 / 19)
    nodes, cls = [np.zeros(d)], [0]
    for lam, q in ((l2, 1), (l3, 2)):
        for k in range(d):
            for sg in (1.0, -1.0):
                x = np.zeros(d)
                x[k] = sg * lam
                nodes.append(x)
                cls.append(q)
    for j, k in itertools.combinations(range(d), 2):
        for sj in (1.0, -1.0):
            for sk in (1.0, -1.0):
                x = np.zeros(d)
                x[j], x[k] = sj * l3, sk * l3
                nodes.append(x)
                cls.append(3)
    for m in range(1 << d):
        nodes.append(np.array([-l5 if (m >> k) & 1 else l5 for k in range(d)]))
        cls.append(4)
    w7 = np.array([(12824 - 9120 * d + 400 * d * d) / 19683, 980 / 6561, (1820 - 400 * d) / 19683, 200 / 19683,
                   6859 / 19683 / 2.0 ** d])
    w5 = np.array([(729 - 950 * d + 50 * d * d) / 729, 245 / 486, (265 - 100 * d) / 1458, 25 / 729, 0.0])
    cls = np.array(cls)
    return [torch.tensor(v, dtype=torch.float64, device="cuda") for v in (np.array(nodes), w7[cls], w5[cls])]


def _gk_rule(d):
    """The same for the tensor 7/15-point Gauss-Kronrod pair: offsets, Kronrod and Gauss weights (of [-1, 1]^d)."""
    P = np.polynomial.legendre
    g, gw = P.leggauss(7)
    q, qw = P.leggauss(16)
    p7 = P.Legendre.basis(7)
    even = [P.Legendre.basis(2 * m) for m in range(5)]
    m = np.array([[np.sum(qw * p7(q) * even[c](q) * q ** k) for c in range(5)] for k in (1, 3, 5, 7)])
    co = np.append(np.linalg.solve(m[:, :4], -m[:, 4]), 1.0)
    e8 = sum(co[c] * even[c] for c in range(5))
    r = np.sort(e8.roots().real)
    for _ in range(3):
        r = r - e8(r) / e8.deriv()(r)
    x = np.sort(np.concatenate([g, r]))
    wk = np.linalg.solve(P.legvander(x, 14).T, np.append(2.0, np.zeros(14)))
    wg = np.zeros(15)
    wg[1::2] = gw
    xs, ks, gs = (torch.tensor(v, dtype=torch.float64, device="cuda") for v in (x, wk, wg))
    i = torch.cartesian_prod(*[torch.arange(15, device="cuda")] * d).reshape(-1, d)
    return xs[i], ks[i].prod(-1), gs[i].prod(-1)


def _exact_rule(case, seed, offsets, w_high, w_low, scale):
    d, n = case["dim"], case["n"]
    c, h = _boxes(d, n, seed, case["kind"] == "gk")
    c, h = c.T.contiguous(), h.T.contiguous()
    a, u = (torch.tensor(v, device="cuda") for v in _params(case, seed))
    vol = torch.prod(h, dim=1) * scale
    high, low = torch.empty_like(vol), torch.empty_like(vol)
    at_once = max(1, int(1.5e8 // (d * len(w_high))))
    for r in range(0, n, at_once):
        x = c[r:r + at_once, None, :] + h[r:r + at_once, None, :] * offsets
        f = _f64(case["family"], a, u, x)
        high[r:r + at_once] = (f * w_high).sum(-1)
        low[r:r + at_once] = (f * w_low).sum(-1)
    err = None if case.get("null") else (vol * high - vol * low).abs()
    return [vol * high, err, torch.prod(2.0 * h, dim=1), None]


def _closed_form(f, a, u):
    """The integral over [0,1]^d."""
    d = len(a)
    if f == G.OSCILLATORY:
        z = complex(math.cos(2 * math.pi * u[0]), math.sin(2 * math.pi * u[0]))
        for v in a:
            z *= (complex(math.cos(v), math.sin(v)) - 1) / (1j * v)
        return z.real
    if f == G.PRODUCT_PEAK:
        return math.prod(p * (math.atan(p * (1 - q)) + math.atan(p * q)) for p, q in zip(a, u))
    if f == G.CORNER_PEAK:
        with localcontext() as ctx:  # an alternating sum that cancels
            ctx.prec = 60
            t = [Decimal(1)]
            sign = [1]
            for v in a:
                t, sign = t + [x + Decimal(float(v)) for x in t], sign + [-x for x in sign]
            s = sum((x / y for x, y in zip(sign, t)), Decimal(0))
            for v in a:
                s /= Decimal(float(v))
            return float(s / math.factorial(d))
    if f == G.GAUSSIAN:
        return math.prod(math.sqrt(math.pi) / (2 * p) * (math.erf(p * (1 - q)) + math.erf(p * q)) for p, q in zip(a, u))
    if f == G.C0:
        return math.prod((2.0 - math.exp(-p * q) - math.exp(-p * (1 - q))) / p for p, q in zip(a, u))
    return math.prod((math.exp(p * min(q, 1.0)) - 1.0) / p for p, q in zip(a, u))


def _exact_grad(case, seed):
    """The Gaussian's integral and its derivatives by a and u."""
    a, u = _grad_rows(case, seed)
    erf = np.vectorize(math.erf)
    p, q = a * (1.0 - u), a * u
    one = math.sqrt(math.pi) / (2.0 * a) * (erf(p) + erf(q))
    ep, eq = np.exp(-p * p), np.exp(-q * q)
    da = -one / a + ((1.0 - u) * ep + u * eq) / a
    du = eq - ep
    v = one.prod(1)
    return [v, v[:, None] / one * da, v[:, None] / one * du]


def _exact_classify(case, seed):
    c, h, i7, err, vf, axis, budget = _classify_inputs(case, seed)
    retire = (err <= budget * vf) | (err <= 50 * 2.0 ** -53 * i7.abs())
    at = torch.nonzero(~retire).squeeze(1)
    on = torch.arange(case["dim"], device="cuda")[:, None] == axis[at].long()[None, :]
    hs = torch.where(on, 0.5 * h[:, at], h[:, at])
    step = torch.where(on, hs, torch.zeros_like(hs))
    zero = torch.zeros_like(i7)
    return {"n_split": None,
            "sums": torch.stack([torch.where(retire, i7, zero).sum(), torch.where(retire, err, zero).sum()]),
            "flags": None, "center": torch.cat([c[:, at] - step, c[:, at] + step], 1),
            "halfw": torch.cat([hs, hs], 1)}


def exact(case, seed):
    k, d = case["kind"], case.get("dim", 0)
    if k == "rule":
        return _exact_rule(case, seed, *_gm_rule(d), 2.0 ** d)
    if k == "gk":
        return _exact_rule(case, seed, *_gk_rule(d), 1.0)
    if k == "autograd":
        return _exact_grad(case, seed)
    if k == "classify":
        return _exact_classify(case, seed)
    if k == "batch":
        of = [(p.family, p.a, p.u) for p in _batch_problems(case, seed)]
    else:
        of = [(FAMILIES[case["family"]], *_params(case, seed))]
    # an adaptive run's error estimate and its counts are no exact values; its integral is
    return {"integral": np.array([_closed_form(*p) for p in of]), "error": None, "counts": None}
