"""Node values from per-axis factors (csrc/gm_factor64.cuh) where they can go
wrong: every dimension around the edges of the leaves and chain parts (d = 3/4:
one leaf of class 5 or two; 8/9: two chain parts or three; 14/15: the cosine's
last dimension with rotations), every lane mapping, and regions whose factors
would over- or underflow (evaluated without factors).

Bounds, per region, against the oracle: 1e-12 of the magnitude of the terms, as
everywhere in these tests; with steep parameters the inner sum S itself is
rounded relative to |S| <= 1100, which moves f by up to |S| 2^-53 per rounding:
16 roundings give 2e-12."""
import numpy as np
import pytest

from paper_2511_01573_gb300 import genz_inputs as G

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

FACTORED = [G.OSCILLATORY, G.PRODUCT_PEAK, G.GAUSSIAN, G.C0, G.DISCONTINUOUS]


def _soa(x):
    return torch.tensor(np.ascontiguousarray(x.T), dtype=torch.float64, device="cuda")


def _check(oracle, gpu_ctx, fam, a, u, c, h, bound):
    outs = [gpu_ctx.eval_rule(fam, a, u, _soa(c), _soa(h), lanes=t) for t in (1, 4, 32, 128)]
    for o in outs[1:]:
        for x, y in zip(outs[0], o):
            assert torch.equal(x, y)
    ref = oracle.rule_regions(fam, a, u, c, h)
    i7, err, vf, ax = (x.cpu().numpy() for x in outs[0])
    assert np.all(np.abs(i7 - ref["i7"]) <= bound * ref["i7abs"])
    assert np.all(np.abs(err - ref["err"]) <= bound * ref["i7abs"])
    clear = ~ref["axis_tie"].astype(bool)
    assert np.array_equal((ax.astype(np.int32) & 0x7F)[clear], ref["axis"][clear])


@pytest.mark.parametrize("fam", FACTORED)
@pytest.mark.parametrize("d", [1, 2, 3, 4, 7, 8, 9, 11, 13, 14, 15])
def test_factored_dimensions(oracle, gpu_ctx, fam, d):
    a, u = G.seed_uniform(7 + d, fam, d, 0.5, 3.0)
    if fam == G.DISCONTINUOUS:
        u = 0.4 + 0.6 * u
    c, h = G.random_boxes(300 + d, 129 if d < 9 else 9, d)
    _check(oracle, gpu_ctx, fam, a, u, c, h, 1e-12)


@pytest.mark.parametrize("fam,scale", [(G.GAUSSIAN, 20.0), (G.GAUSSIAN, 400.0), (G.C0, 300.0),
                                       (G.DISCONTINUOUS, 90.0), (G.PRODUCT_PEAK, 1e40)])
@pytest.mark.parametrize("d", [1, 5, 9])
def test_factors_without_exponent_room(oracle, gpu_ctx, fam, scale, d):
    a, u = G.seed_uniform(5 + d, fam, d, 0.5 * scale, scale)
    if fam == G.DISCONTINUOUS:
        u = 0.4 + 0.6 * u
        a[::2] = -a[::2]  # the inner sum cancels: factors far apart, f moderate
    c, h = G.random_boxes(400 + d, 131 if d < 9 else 11, d)
    # the whole domain as well: the widest spread of factors
    c, h = np.concatenate([c, np.full((1, d), 0.5)]), np.concatenate([h, np.full((1, d), 0.5)])
    _check(oracle, gpu_ctx, fam, a, u, c, h, 3e-12)


@pytest.mark.parametrize("fam,scale", [(G.GAUSSIAN, 1.0), (G.GAUSSIAN, 60.0), (G.C0, 1.0),
                                       (G.C0, 300.0), (G.DISCONTINUOUS, 1.0),
                                       (G.PRODUCT_PEAK, 1.0)])
@pytest.mark.parametrize("d,n", [(1, 5), (2, 33), (3, 6), (4, 3), (5, 1)])
def test_gauss_kronrod_factors(oracle, gpu_ctx, fam, scale, d, n):
    """The Gauss-Kronrod rule from per-axis factors: a warp per region up to
    d = 3, a block from d = 4, with and without exponent room."""
    a, u = G.seed_uniform(17 + d, fam, d, 0.5 * scale, 3.0 * scale)
    if fam == G.DISCONTINUOUS:
        u = 0.4 + 0.6 * u
    c, h = G.random_boxes(800 + d, n, d)
    c, h = np.concatenate([c, np.full((1, d), 0.5)]), np.concatenate([h, np.full((1, d), 0.5)])
    ref = oracle.rule_gk_regions(fam, a, u, c, h)
    ik, err, vf, ax = (x.cpu().numpy() for x in gpu_ctx.eval_rule_gk(fam, a, u, _soa(c), _soa(h)))
    assert np.all(np.abs(ik - ref["ik"]) <= 1e-12 * ref["scale"] + 1e-300)
    assert np.all(np.abs(err - ref["err"]) <= 1e-12 * ref["scale"] + 1e-300)
    clear = ~ref["axis_tie"].astype(bool)
    assert np.array_equal((ax.astype(np.int32) & 0x7F)[clear], ref["axis"][clear])


@pytest.mark.parametrize("fam,scale", [(G.GAUSSIAN, 1.0), (G.GAUSSIAN, 60.0), (G.C0, 1.0),
                                       (G.C0, 300.0), (G.DISCONTINUOUS, 1.0),
                                       (G.PRODUCT_PEAK, 1.0)])
@pytest.mark.parametrize("d,n", [(1, 65), (2, 64), (3, 63), (8, 9), (9, 7)])
def test_adjoint_factors(oracle, gpu_ctx, fam, scale, d, n):
    """gmq_rule_grad from per-axis factors, with and without exponent room: the
    bounds of the adjoint tests (1e-12 of the largest component), and three of
    them for steep parameters, as above."""
    a, u = G.seed_uniform(19 + d, fam, d, 0.5 * scale, 3.0 * scale)
    if fam == G.DISCONTINUOUS:
        u = 0.4 + 0.6 * u
    c, h = G.random_boxes(900 + d, n, d)
    go, qo = oracle.rule_grad(fam, a, u, c, h)
    g, q = gpu_ctx.rule_grad(fam, a, u, _soa(c), _soa(h))
    scale_g = np.max(np.abs(go)) + abs(qo)
    bound = 1e-12 if scale == 1.0 else 3e-12
    assert abs(q - qo) <= bound * scale_g
    assert np.all(np.abs(np.asarray(g) - go) <= bound * scale_g)
