"""The mixed form's tree walk (csrc/gm_region32.cuh, one lane, 3 <= d <= 12)
against the node-by-node kernel (32 lanes): both evaluate every node with the
same FP32 operations, so split axes are equal, and rule values differ only by
the compensated sums' rounding: at most 2^-24 of a compensation that is at most
n 2^-25 of the class sum, for each of n <= 4409 nodes, i.e. below n^2 2^-49 =
3.5e-8 of the magnitude of the terms in the worst case and n 2^-49 = 8e-12 for
roundings of random sign, which is what is asked.  Parameters reach past the
fast forms of the reciprocal and the cosine."""
import numpy as np
import pytest

from paper_2511_01573_gb300 import genz_inputs as G

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _soa(x):
    return torch.tensor(np.ascontiguousarray(x.T), dtype=torch.float64, device="cuda")


@pytest.mark.parametrize("fam,scale", [(f, 1.0) for f in range(7)] +
                         [(G.PRODUCT_PEAK, 1e-8), (G.PRODUCT_PEAK, 1e6), (G.CORNER_PEAK, 1e9),
                          (G.OSCILLATORY, 3e4)])
@pytest.mark.parametrize("d,n", [(3, 129), (4, 33), (5, 65), (8, 31), (11, 5), (12, 3)])
def test_walk_against_node_by_node(oracle, gpu_ctx, fam, scale, d, n):
    from paper_2511_01573_gb300 import gmq
    a, u = G.seed_uniform(23 + d, fam, d, 0.5 * scale, 3.0 * scale)
    if fam == G.DISCONTINUOUS:
        u = 0.4 + 0.6 * u
    c, h = G.random_boxes(950 + d, n, d)
    walk, flat = ([x.cpu().numpy() for x in
                   gpu_ctx.eval_rule(fam, a, u, _soa(c), _soa(h), precision=gmq.MIXED, lanes=t)]
                  for t in (1, 32))
    terms = oracle.rule_regions(fam, a, u, c, h)["i7abs"]
    for x, y in zip(walk[:2], flat[:2]):
        fine = np.isfinite(y)
        assert np.array_equal(fine, np.isfinite(x))
        assert np.all(np.abs(x - y)[fine] <= 8e-12 * np.maximum(terms, np.abs(y))[fine])
    assert np.array_equal(walk[2], flat[2])
    assert np.array_equal(walk[3], flat[3])
