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
