"""The density factor x1^a x2^a (1-x1)^b (1-x2)^b of the global weights over its forms: products for b = 0..3, an
exponential for others, CUDA's powers at the ends of the range.  One channel with J = P = alpha = 1, so that
the weight is the factor; the reference is the formula in extended precision, and the factor carries at most 16
roundings (logarithms good to 2^-60, one exponential each, a handful of products)."""
import numpy as np
import pytest

from paper_2602_06895_gb300 import ps

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("a", [-1.1, 0.0, 0.5, -0.3])
@pytest.mark.parametrize("b", [0.0, 1.0, 2.0, 3.0, 2.5, 4.7])
def test_density_factor(a, b):
    import torch

    from paper_2602_06895_gb300 import build

    build.build()
    g = np.random.default_rng(3)
    n = 20000
    x1, x2 = 10.0 ** g.uniform(-9, 0, n), g.random(n)
    x1[:6] = 0.5, 1.0 - 2.0 ** -53, 2.0 ** -300, 1e-310, 0.25, 1.0
    x2[:6] = 1.0 - 2.0 ** -52, 0.5, 0.75, 0.5, 1e-12, 0.5
    one = torch.ones((1, n), dtype=torch.float64, device="cuda")
    w = torch.empty(n, dtype=torch.float64, device="cuda")
    t1, t2 = (torch.tensor(x, device="cuda") for x in (x1, x2))
    ps.global_weights(one, [1.0], w, P=one, x1=t1, x2=t2, pdf=(a, b))
    torch.cuda.synchronize()
    X1, X2 = np.longdouble(x1), np.longdouble(x2)
    A, B = np.longdouble(a), np.longdouble(b)
    ref = X1 ** A * X2 ** A * (1 - X1) ** B * (1 - X2) ** B
    got = w.cpu().numpy()
    over = ref > np.finfo(np.float64).max  # a subnormal x to a negative power: beyond double
    assert np.all(np.isinf(got[over]))
    got, ref = got[~over], ref[~over]
    assert np.all(np.abs(got - ref) <= 16 * 2.0 ** -53 * 2 * ref + 1e-320)
