"""The Jacobian of the Breit-Wigner map over all three of its angle regions: J = D M Gamma (1 + tan^2 u), u = atan a + D r,
in 113-bit arithmetic from the kernel's own M^2 and M Gamma.

Bound: a and b carry 3 roundings each, D = atan2(b - a, 1 + a b) 10 (its derivative in either argument is at most 1
relative to D).  In the outer regions the angle from the nearer end carries 12, its tangent 1.6 times those (at most
pi/4), the reciprocal of 1 -+ a T 22, squared 44, 1 + T^2 and 1 + a^2 19 and 5: 85 in all.  In the middle u is a sum of
two angles up to pi/2, 30 roundings absolute, and 1 + T^2 twice that: 75 with D.  128 are allowed."""
import numpy as np
import pytest

from test_gpu_fp64_ops import EPS, LD, run_op, torch_cuda  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M, G", [(80.4, 2.1), (125.0, 0.004), (173.0, 1.4), (1.0, 3.0)])
@pytest.mark.parametrize("jit", [False, True], ids=["interpreter", "compiled"])
def test_breit_wigner_jacobian(torch_cuda, M, G, jit):  # noqa: F811
    if np.finfo(LD).eps > 2.0 ** -100:
        pytest.skip("needs a long double of 113 bits")
    rng = np.random.default_rng(13)
    n = 6000
    r = rng.random(n)
    r[:3] = 0.0, 1.0, 0.5
    kind = rng.random(n)
    lo = np.where(kind < 0.3, 0.0, 10.0 ** rng.uniform(-6, 5, n))
    lo = np.where(kind > 0.7, np.maximum(0.0, M * M - M * G * rng.uniform(-5, 50, n)), lo)  # about the peak
    hi = lo + np.where(rng.random(n) < 0.5, 10.0 ** rng.uniform(-3, 8, n), M * G * rng.uniform(0.1, 100, n))
    x, jac = run_op(torch_cuda, "INVARIANT_BW", [0, M, G, 1, 2], 2, [r, lo, hi], jit)
    mg, m2 = LD(M * G), LD(M * M)
    a, b = (LD(lo) - m2) / mg, (LD(hi) - m2) / mg
    D = np.arctan2((LD(hi) - LD(lo)) / mg, 1 + a * b)
    u = np.arctan(a) + D * LD(r)
    ref = D * mg * (1 + np.tan(u) ** 2)
    assert np.all(np.abs(LD(jac) - ref) <= 128 * EPS * ref)
    assert np.all((x >= lo) & (x <= hi))
