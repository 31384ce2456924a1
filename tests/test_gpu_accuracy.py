"""Accuracy of the FP64 rules against long double arithmetic (113 bits on the
GPU's Arm host, 64 on x86), over slopes, dimensions and boxes at which the
per-axis and fixed-point forms have to hold bits that random boxes of moderate
slopes do not ask for.  Units: eps = 2^-53, half the spacing of doubles at 1."""
import numpy as np
import pytest

from paper_2511_01573_gb300 import genz_inputs as G

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

LD = np.longdouble
EPS = 2.0 ** -53


def _soa(x):
    return torch.tensor(np.ascontiguousarray(x.T), dtype=torch.float64, device="cuda")


@pytest.mark.parametrize("lanes", [1, 32])
def test_cosine_factors_at_the_ends_of_the_reduction(gpu_ctx, lanes):
    """cos(x) of the cosine's centre factor at odd multiples of pi / 256, where the
    reduced argument is largest, and where |cos| < 1/2, so that the sine's part of
    it weighs: a region of width 2^-40 around x in d = 1 has I7 / (2 h) = cos(x) to
    2^-80.  The sine and the cosine are within 1.2 eps; the rule's five products
    and sums, relative to |cos| < 1/2, add half of up to 2 eps: 2.2 eps."""
    k = np.arange(1, 1303, 2)
    x = np.concatenate([k * np.pi / 256 + t for t in (-1e-6, -1e-9, 1e-9, 1e-6)])
    x = x[np.abs(np.cos(x)) < 0.5]
    h = np.full((len(x), 1), 2.0 ** -40)
    i7 = gpu_ctx.eval_rule(G.OSCILLATORY, np.ones(1), np.zeros(1), _soa(x[:, None]), _soa(h),
                           lanes=lanes)[0].cpu().numpy()
    err = np.abs((i7 * 2.0 ** 39).astype(LD) - np.cos(x.astype(LD)))
    assert np.max(err) <= 2.2 * EPS


def _factor(fam, a, u, b, x):
    """One axis' factor of f in long double (a scalar's worth of the family)."""
    t = x - u
    if fam == G.GAUSSIAN:
        return np.exp(-b * t * t)
    if fam == G.C0:
        return np.exp(-a * np.abs(t))
    if fam == G.PRODUCT_PEAK:
        return 1 / (t * t + b)
    return np.where(t > 0, LD(0), np.exp(a * x))


def _exact_i7(fam, a, u, c, h):
    """The degree-7 rule's value on one region and the sum of its terms'
    magnitudes, unit volume, in long double: class sums of products of factors, with
    the generators and weights that the rule has, rounded to FP64."""
    d = len(a)
    a, u, c, h = (np.asarray(v, dtype=LD) for v in (a, u, c, h))
    b = (1 / (a * a) if fam == G.PRODUCT_PEAK else a * a).astype(np.float64).astype(LD)
    l2, l3, l5 = (LD(np.sqrt(v)) for v in (9 / 70, 9 / 10, 9 / 19))
    f = lambda lam: _factor(fam, a, u, b, c + lam * h)
    f0 = f(LD(0))
    p = [f(l) + f(-l) for l in (l2, l3, l5)]
    others = [np.prod(np.delete(f0, k)) for k in range(d)]
    s4 = LD(0)
    for j in range(d):
        for k in range(j + 1, d):
            s4 += p[1][j] * p[1][k] * np.prod(np.delete(f0, [j, k]))
    s = [np.prod(f0), sum(o * v for o, v in zip(others, p[0])),
         sum(o * v for o, v in zip(others, p[1])), s4, np.prod(p[2])]
    w = [LD(v / 19683) for v in (12824 - 9120 * d + 400 * d * d, 2940, 1820 - 400 * d, 200,
                                 6859 / 2 ** d)]
    return sum(x * y for x, y in zip(w, s)), sum(abs(x * y) for x, y in zip(w, s))


def _cases(fam, d, n, lo, hi, whole, seed):
    rng = np.random.default_rng(seed)
    for _ in range(n):
        a, u = rng.uniform(lo, hi, d), rng.uniform(0, 1, d)
        if fam == G.DISCONTINUOUS:
            u = 0.4 + 0.6 * u
        x = rng.uniform(0, 1, (2, d))
        c, h = 0.5 * (x[0] + x[1]), 0.5 * np.abs(x[0] - x[1])
        if whole:
            c, h = np.full(d, 0.5), np.full(d, 0.5)
        yield a, u, c, h


def _rms_errors(gpu_ctx, fam, cases, exact):
    """rms over the cases of I7's error relative to its terms: the default form's
    and the node-wise form's."""
    from paper_2511_01573_gb300 import gmq
    out = np.zeros(2)
    n = 0
    for a, u, c, h in cases:
        ref, terms = exact(fam, a, u, c, h)
        if terms == 0:
            continue
        vol = np.prod((2 * h).astype(LD))
        for i, mode in enumerate((gmq.EVAL_SEPARABLE, gmq.EVAL_NODEWISE)):
            gpu_ctx.set_eval_mode(mode)
            try:
                i7 = gpu_ctx.eval_rule(fam, a, u, _soa(c[None]), _soa(h[None]), lanes=32)[0]
            finally:
                gpu_ctx.set_eval_mode(gmq.EVAL_SEPARABLE)
            out[i] += float((LD(i7.item()) / vol - ref) / terms) ** 2
        n += 1
    return np.sqrt(out / n)


@pytest.mark.parametrize("whole", [False, True])
@pytest.mark.parametrize("fam,lo,hi,d", [(G.C0, 4, 12, 4), (G.C0, 4, 12, 8), (G.C0, 20, 60, 8),
                                         (G.C0, 0.5, 3, 5), (G.GAUSSIAN, 5, 15, 4),
                                         (G.GAUSSIAN, 0.5, 3, 6), (G.GAUSSIAN, 5, 15, 8),
                                         (G.DISCONTINUOUS, 5, 15, 6)])
def test_steep_factors(gpu_ctx, fam, lo, hi, d, whole):
    """Factors far from 1: the difference that a factor is the exponential of is
    kept to 2^-57 (2^-53 where it is 15 and more), not rounded relative to its own
    size, so that products of factors are as near as the node-wise form, which
    rounds every node's inner sum, small where f is large: at most 1.25 of its
    error, and half an eps for the products' own roundings."""
    mine, node = _rms_errors(gpu_ctx, fam, _cases(fam, d, 48, lo, hi, whole, 11 * d + int(lo)),
                             _exact_i7)
    assert mine <= 1.25 * node + 0.5 * EPS


@pytest.mark.parametrize("fam,lo,hi,d", [(G.GAUSSIAN, 2.8, 3.2, 12), (G.GAUSSIAN, 2.8, 3.2, 14),
                                         (G.GAUSSIAN, 0.5, 3, 14), (G.GAUSSIAN, 2.8, 3.2, 16),
                                         (G.PRODUCT_PEAK, 4.5, 5.5, 14),
                                         (G.PRODUCT_PEAK, 4.5, 5.5, 16),
                                         (G.PRODUCT_PEAK, 10, 60, 16), (G.C0, 4, 12, 14)])
def test_class_sums_of_many_products(gpu_ctx, fam, lo, hi, d):
    """2^12 and more products of tables whose largest entries dominate (the whole
    domain): the sums of integer products are exact but for the tables' entries,
    each within half an eps of its table's largest, so the node-wise form's error
    is met up to a quarter and half an eps."""
    mine, node = _rms_errors(gpu_ctx, fam, _cases(fam, d, 24, lo, hi, True, d), _exact_i7)
    assert mine <= 1.25 * node + 0.5 * EPS


@pytest.mark.parametrize("fam,lo,hi", [(G.PRODUCT_PEAK, 10, 20), (G.PRODUCT_PEAK, 30, 60),
                                       (G.PRODUCT_PEAK, 100, 300), (G.C0, 5, 20), (G.C0, 0.5, 3),
                                       (G.GAUSSIAN, 3, 9)])
@pytest.mark.parametrize("d", [1, 2, 3, 4, 5, 6])
def test_gauss_kronrod_far_factors(gpu_ctx, oracle, fam, lo, hi, d):
    """I_K of the tensor rule on the whole domain, where a few of the 15^d terms
    make the sum: the product over the axes of the sums of 15 terms in long
    double.  A factor is within 1.5 eps, the centre within 2, the entries of axis
    0 within half an eps of its largest, row products and sums below: 1.5 sqrt(d) +
    4 eps rms, and the coordinates' rounding, half an eps of |x - u| <= 1, which
    moves f by a for the exponentials and, worst, by 2 a^2 |x - u| <= a for the
    peak, times sqrt(d)."""
    K = np.asarray(oracle.gk_table())
    rng = np.random.default_rng(100 * d + int(lo))
    sq = []
    for _ in range(12):
        a, u = rng.uniform(lo, hi, d), rng.uniform(0, 1, d)
        if fam == G.GAUSSIAN:
            u = 0.25 + 0.5 * u
        la, lu = a.astype(LD), u.astype(LD)
        b = (1 / (la * la) if fam == G.PRODUCT_PEAK else la * la).astype(np.float64).astype(LD)
        from paper_2511_01573_gb300 import gmq
        T = np.asarray(gmq.gk_table()).astype(LD)
        x = LD(0.5) + LD(0.5) * T[:15]
        ref = LD(1)
        for k in range(d):
            ref *= np.sum(T[15:30] * _factor(fam, la[k], lu[k], b[k], x)) / 2
        half = _soa(np.full((1, d), 0.5))
        ik = gpu_ctx.eval_rule_gk(fam, a, u, half, half)[0].item()
        sq.append(float((LD(ik) - ref) / ref) ** 2)
    assert np.sqrt(np.mean(sq)) <= (1.5 * d ** 0.5 + 4 + 0.5 * d ** 0.5 * hi / 4) * EPS


def _exact_corner(fam, a, u, c, h):
    d = len(a)
    a, c, h = (np.asarray(v, dtype=LD) for v in (a, c, h))
    l2, l3, l5 = (LD(np.sqrt(v)) for v in (9 / 70, 9 / 10, 9 / 19))
    s0, ah = 1 + np.sum(a * c), a * h
    f = lambda s: 1 / s ** (d + 1)
    s4 = LD(0)
    for j in range(d):
        for k in range(j + 1, d):
            for sj in (1, -1):
                for sk in (1, -1):
                    s4 += f(s0 + l3 * (sj * ah[j] + sk * ah[k]))
    s = np.array([s0], dtype=LD)
    for k in range(d):
        s = np.concatenate([s + l5 * ah[k], s - l5 * ah[k]])
    S = [f(s0), np.sum(f(s0 + l2 * ah) + f(s0 - l2 * ah)), np.sum(f(s0 + l3 * ah) + f(s0 - l3 * ah)),
         s4, np.sum(f(s))]
    w = [LD(v / 19683) for v in (12824 - 9120 * d + 400 * d * d, 2940, 1820 - 400 * d, 200,
                                 6859 / 2 ** d)]
    return sum(x * y for x, y in zip(w, S)), sum(abs(x * y) for x, y in zip(w, S))


@pytest.mark.parametrize("d,total", [(4, 3.3), (8, 2.4), (8, 3.3), (12, 1.85), (12, 3.3),
                                     (14, 2.4), (14, 3.3), (16, 1.2), (16, 2.4), (16, 3.3)])
def test_corner_powers(gpu_ctx, d, total):
    """The corner peak on the whole domain, S spanning up to a factor of almost 4,
    whose powers d + 1 lie up to 2^34 apart: at most the node-wise form's error and
    half an eps."""
    def cases():
        rng = np.random.default_rng(d)
        for _ in range(24 if d < 14 else 8):
            a = rng.uniform(0.1, 1.0, d)
            yield a * (total / a.sum()), np.zeros(d), np.full(d, 0.5), np.full(d, 0.5)
    mine, node = _rms_errors(gpu_ctx, G.CORNER_PEAK, cases(), _exact_corner)
    assert mine <= node + 0.5 * EPS


@pytest.mark.parametrize("lanes", [1, 32])
def test_cosine_from_sixteen_on(gpu_ctx, lanes):
    """The same for arguments in units of 2^-54 (16 <= |x| < 256: within 1.4 eps) and
    on both sides of the two limits."""
    rng = np.random.default_rng(5)
    x = np.concatenate([np.arange(1305, 20861, 2) * np.pi / 256 + 1e-7, rng.uniform(16, 256, 4000),
                        16 + np.arange(-8, 9) * 2.0 ** -49, 256 + np.arange(-8, 9) * 2.0 ** -45])
    x = x[np.abs(np.cos(x)) < 0.5]
    h = np.full((len(x), 1), 2.0 ** -40)
    i7 = gpu_ctx.eval_rule(G.OSCILLATORY, np.ones(1), np.zeros(1), _soa(x[:, None]), _soa(h),
                           lanes=lanes)[0].cpu().numpy()
    err = np.abs((i7 * 2.0 ** 39).astype(LD) - np.cos(x.astype(LD)))
    assert np.max(err) <= 2.4 * EPS


@pytest.mark.parametrize("fam,lo,hi", [(G.GAUSSIAN, 0.5, 3), (G.C0, 0.5, 3),
                                       (G.PRODUCT_PEAK, 2, 6)])
def test_mean_error_of_table_roundings(gpu_ctx, fam, lo, hi):
    """Entries of the integer tables lose the one or two bits by which they are below
    their table's largest, so that ties are common: rounded up they would move a
    class sum by up to an eps and I7 by 0.15 of one in the mean.  Errors of 960
    regions of rms 0.4 eps have a mean within 0.04 (three standard deviations) of
    their expectation, for which the other roundings, to nearest, leave 0.06."""
    rng = np.random.default_rng(3)
    d, err = 6, []
    for _ in range(60):
        a = rng.uniform(lo, hi, d)
        u = np.floor(rng.uniform(0, 1, d) * 1024) / 1024  # c - u is exact
        q = rng.integers(0, 3, (16, d))
        h = 2.0 ** -(q + 1.0)
        c = (2 * np.floor(rng.uniform(0, 1, (16, d)) * 2.0 ** q) + 1) * h
        i7 = gpu_ctx.eval_rule(fam, a, u, _soa(c), _soa(h))[0].cpu().numpy()
        for i in range(16):
            ref, terms = _exact_i7(fam, a, u, c[i], h[i])
            err.append(float((LD(i7[i]) / np.prod((2 * h[i]).astype(LD)) - ref) / terms) / EPS)
    assert abs(np.mean(err)) <= 0.1


@pytest.mark.parametrize("lanes", [1, 4, 32])
@pytest.mark.parametrize("d", [3, 6, 12])
def test_mixed_flagged_region_with_a_slope_beyond_fp32(gpu_ctx, lanes, d):
    """A region above the discontinuous integrand's threshold on its first axis is 0,
    whatever the slopes on the axes after it."""
    from paper_2511_01573_gb300 import gmq
    a, u = np.ones(d), np.full(d, 2.0)
    a[1:], u[0] = 1e39, -1.0
    c = np.random.default_rng(d).uniform(0.3, 0.7, (9, d))
    i7, err, _, _ = gpu_ctx.eval_rule(G.DISCONTINUOUS, a, u, _soa(c), _soa(np.full((9, d), 0.1)),
                                      precision=gmq.MIXED, lanes=lanes)
    assert torch.all(i7 == 0.0) and torch.all(err == 0.0)


def _exact_cosine(fam, a, u, c, h):
    d = len(a)
    c0 = LD(2.0 * np.pi * u[0])
    a, c, h = (np.asarray(v, dtype=LD) for v in (a, c, h))
    f0 = np.cos(c0 + np.sum(a * c))
    z = [2 * np.cos(LD(np.sqrt(v)) * a * h) for v in (9 / 70, 9 / 10, 9 / 19)]
    s4 = (np.sum(z[1]) ** 2 - np.sum(z[1] ** 2)) / 2
    s = [LD(1), np.sum(z[0]), np.sum(z[1]), s4, np.prod(z[2])]
    n = [1, 2 * d, 2 * d, 2 * d * (d - 1), 2 ** d]
    w = [LD(v / 19683) for v in (12824 - 9120 * d + 400 * d * d, 2940, 1820 - 400 * d, 200,
                                 6859 / 2 ** d)]
    return f0 * sum(x * y for x, y in zip(w, s)), sum(abs(x) * y for x, y in zip(w, n))


@pytest.mark.parametrize("whole", [False, True])
@pytest.mark.parametrize("lo,hi,d", [(5, 15, 4), (5, 15, 8), (5, 15, 14), (30, 90, 3), (0.5, 3, 6)])
def test_steep_cosine(gpu_ctx, lo, hi, d, whole):
    """Angles and the centre's sum in fixed point, half a unit of 2^-57 each: what is
    left is the roundings of the products, below half an eps of the terms, whatever
    the sum's size, which the node-wise form's error grows with."""
    mine, node = _rms_errors(gpu_ctx, G.OSCILLATORY, _cases(G.OSCILLATORY, d, 48, lo, hi, whole, d),
                             _exact_cosine)
    assert mine <= 0.5 * EPS + 0.25 * node
