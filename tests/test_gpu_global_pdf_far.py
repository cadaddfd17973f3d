"""The density factor of the global weights where its logarithm is beyond 600, out of the short exponential's range: a
product there carries the rounding of an argument of up to 709, 2^-44, unless the argument's rest goes along.  The bound
is that of test_gpu_global_pdf.py, 16 roundings."""
import numpy as np
import pytest

from paper_2602_06895_gb300 import ps
from test_gpu_flow import torch_cuda  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("a, b", [(-3.0, 2.0), (-3.1, 0.0), (2.9, 2.5), (3.0, 1.0), (-700.0, 3.0), (0.0, 400.0), (0.5, 350.5)])
def test_far_density_factor(torch_cuda, a, b):  # noqa: F811
    torch = torch_cuda
    g = np.random.default_rng(5)
    n = 20000
    # a log(x1 x2) and b log((1 - x1)(1 - x2)) over -700 .. 700
    scale = 700.0 / abs(a if abs(a) > abs(b) else b)
    x1 = np.exp(-scale * g.uniform(0.4, 0.99, n)) if abs(a) > abs(b) else -np.expm1(-scale * g.uniform(0.4, 0.99, n))
    x2 = 0.5 * g.random(n) ** 2 + 1e-3 if abs(a) < 100 else 1.0 - 1e-4 * g.random(n)
    one = torch.ones((1, n), dtype=torch.float64, device="cuda")
    w = torch.empty(n, dtype=torch.float64, device="cuda")
    t1, t2 = (torch.tensor(x, device="cuda") for x in (x1, x2))
    ps.global_weights(one, [1.0], w, P=one, x1=t1, x2=t2, pdf=(a, b))
    got = w.cpu().numpy()
    X1, X2, A, B = np.longdouble(x1), np.longdouble(x2), np.longdouble(a), np.longdouble(b)
    if np.finfo(np.longdouble).eps > 2.0 ** -70:  # no quad arithmetic: powers of 64-bit extended numbers lose 10 bits
        pytest.skip("needs a long double of more than 64 bits")
    # the powers are of the double 1 - x: its own rounding, b/2 ulps of the factor, is the argument's
    ref = X1 ** A * X2 ** A * np.longdouble(1.0 - x1) ** B * np.longdouble(1.0 - x2) ** B
    fin = (ref < 1.7e308) & (ref > 1e-300)
    assert fin.sum() > n // 4
    assert np.all(np.abs(got[fin] - ref[fin]) <= 16 * 2.0 ** -53 * 2 * ref[fin])
