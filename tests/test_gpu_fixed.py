"""The corner peak in fixed point (csrc/gm_fixed64.cuh) where it can go wrong:
dimensions around the chain parts' edges and every exponent d + 1 form, regions
at the limits of the scaling (S spanning almost a factor of 4, small and large
S), and regions it hands to the separable form (wider spans, S near or below
zero), for every lane mapping.

Bounds, per region, against the oracle: 1e-12 of the magnitude of the terms.
The fixed-point form is within (d + 1) 2^-57 of the exact node values; the
oracle's own chain of d + 1 roundings and a power moves f by up to (d + 1) (d +
3) 2^-53 = 4e-14 at d = 16."""
import numpy as np
import pytest

from paper_2511_01573_gb300 import genz_inputs as G

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _soa(x):
    return torch.tensor(np.ascontiguousarray(x.T), dtype=torch.float64, device="cuda")


def _check(oracle, gpu_ctx, a, c, h, bound=1e-12):
    u = np.zeros_like(a)
    outs = [gpu_ctx.eval_rule(G.CORNER_PEAK, a, u, _soa(c), _soa(h), lanes=t)
            for t in (1, 4, 32, 128)]
    for o in outs[1:]:
        for x, y in zip(outs[0], o):
            assert torch.equal(x, y)
    ref = oracle.rule_regions(G.CORNER_PEAK, a, u, c, h)
    i7, err, vf, ax = (x.cpu().numpy() for x in outs[0])
    assert np.all(np.abs(i7 - ref["i7"]) <= bound * ref["i7abs"])
    assert np.all(np.abs(err - ref["err"]) <= bound * ref["i7abs"])
    clear = ~ref["axis_tie"].astype(bool)
    assert np.array_equal((ax.astype(np.int32) & 0x7F)[clear], ref["axis"][clear])


@pytest.mark.parametrize("d", [1, 2, 3, 4, 5, 7, 8, 9, 11, 12, 15, 16])
def test_corner_dimensions(oracle, gpu_ctx, d):
    a, _ = G.seed_genz(3 + d, G.CORNER_PEAK, d, 1.85)
    c, h = G.random_boxes(500 + d, {1: 400, 16: 2, 15: 3}.get(d, 131 if d < 9 else 9), d)
    _check(oracle, gpu_ctx, a, c, h)


@pytest.mark.parametrize("total", [0.01, 1.2, 1.6, 2.4, 40.0, 3e11])
@pytest.mark.parametrize("d", [2, 6, 10])
def test_corner_spans(oracle, gpu_ctx, total, d):
    # whole-domain boxes: S spans (1, 1 + total) times lambda3's share
    a, _ = G.seed_genz(9 + d, G.CORNER_PEAK, d, total)
    c, h = G.random_boxes(600 + d, 40, d)
    c = np.concatenate([c, np.full((2, d), 0.5)])
    h = np.concatenate([h, np.full((1, d), 0.5), np.full((1, d), 0.25)])
    _check(oracle, gpu_ctx, a, c, h)


@pytest.mark.parametrize("d", [3, 8])
def test_corner_small_and_negative_sums(oracle, gpu_ctx, d):
    # a < 0: S falls from 1 towards zero and below it over the domain; boxes
    # whose node sums come within 1e-2 of zero are left out (f is singular)
    a = -G.seed_genz(4 + d, G.CORNER_PEAK, d, 2.0)[0]
    c, h = G.random_boxes(700 + d, 400, d)
    s, r = 1.0 + c @ a, h @ np.abs(a)
    keep = (s - r > 1e-2) | (s + r < -1e-2)
    c, h = c[keep], h[keep]
    assert np.any(s[keep] < 0) and np.any(s[keep] > 0)
    # S comes from a cancelling sum: its rounding, 2^-53 per term, is up to
    # (d + 1) d 2^-53 / 1e-2 of f
    _check(oracle, gpu_ctx, a, c, h, 1e-12 + (d + 1) * (d + 1) * 2.0 ** -52 / 1e-2)
