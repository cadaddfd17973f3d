"""Single FP64 ops of the map kernels (one-instruction graphs through the C ABI, interpreted and
compiled) on arguments at the edges of their short forms: exponents, zeros, infinities and NaN for the
division and the root, bounds and exponents of every branch of the power-law map, both ends of the
Breit-Wigner angle.  References are the formulas in extended precision (np.longdouble); tolerances are
counted in roundings, eps = 2^-52."""
import numpy as np
import pytest

from paper_2602_06895_gb300 import ps

pytestmark = pytest.mark.gpu

EPS = 2.0 ** -52
LD = np.longdouble


@pytest.fixture(scope="module")
def torch_cuda():
    import torch

    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2602_06895_gb300 import build

    build.build()
    return torch


def run_op(torch, op, args, n_out, cols, jit):
    """Outputs (first two) of one op on the columns `cols` (float64 arrays), args as for Graph.add."""
    g = ps.Graph.create(len(cols))
    o = g.add(op, args, n_out)
    one = g.add("MUL", [0.0, 0], 1)[0] if n_out < 2 else None
    g.set_outputs([o[0], o[1] if n_out > 1 else one, o[0]], [ps.ROLE_X1, ps.ROLE_X2, ps.ROLE_WEIGHT])
    prog = ps.Program([g], jit=jit)
    r = torch.tensor(np.stack(cols), device="cuda")
    out, ws = prog.alloc([r.shape[1]], 0)
    prog.map(0, r, out, ws)
    torch.cuda.synchronize()
    return out["x1"].cpu().numpy(), out["x2"].cpu().numpy()


SPECIAL = [0.0, -0.0, 1.0, -1.0, 0.5, 2.0, 2.0 - EPS, 1.0 + EPS, 4.0 - 4 * EPS, 3.0, 1e-310, 5e-324, -1e-310, 2.2250738585072014e-308,
           1.7976931348623157e308, -1.7976931348623157e308, 1e-290, 1e290, 1e200, 1e-200, np.inf, -np.inf, np.nan]


@pytest.mark.parametrize("jit", [False, True], ids=["interpreter", "compiled"])
def test_division_and_root(torch_cuda, jit):
    rng = np.random.default_rng(5)
    a, b = (x.ravel() for x in np.meshgrid(SPECIAL, SPECIAL))
    m = np.exp2(rng.uniform(-300, 300, 20000)) * rng.choice([-1.0, 1.0], 20000)
    a, b = np.concatenate([a, m]), np.concatenate([b, m[::-1]])
    with np.errstate(all="ignore"):
        ref, root = a / b, np.sqrt(np.abs(a))
    q, _ = run_op(torch_cuda, "DIV", [0, 1], 1, [a, b], jit)
    s, _ = run_op(torch_cuda, "SQRT", [0], 1, [np.abs(a)], jit)
    for got, want in ((q, ref), (s, root)):
        fin = np.isfinite(want)
        assert np.array_equal(np.isnan(got), np.isnan(want))
        assert np.array_equal(got[~fin & ~np.isnan(want)], want[~fin & ~np.isnan(want)])
        # half an ulp and a little: the correctly rounded value or its neighbour
        assert np.all(np.abs(got[fin] - want[fin]) <= np.spacing(np.abs(want[fin])))
        assert np.mean(got[fin] == want[fin]) > 0.999


@pytest.mark.parametrize("nu", [0.0, 0.3, 0.5, 2.0 / 3.0, 0.75, 0.8, 5.0 / 6.0, 0.9, 1.0, 1.4])
@pytest.mark.parametrize("jit", [False, True], ids=["interpreter", "compiled"])
def test_power_law_map(torch_cuda, nu, jit):
    rng = np.random.default_rng(7)
    n, a = 6000, 1e-4
    r = rng.random(n)
    r[:3] = 0.0, 1.0, 0.5
    lo = np.where(rng.random(n) < 0.4, 0.0, 10.0 ** rng.uniform(-8, 6, n))
    hi = lo + 10.0 ** rng.uniform(-12, 8, n) * rng.choice([1.0, 1e-6], n)
    hi[3:6] = lo[3:6]  # an empty range
    x, jac = run_op(torch_cuda, "INVARIANT_NU", [0, 0.0, nu, 1, 2, a], 2, [r, lo, hi], jit)
    R, X0, X1, A = LD(r), LD(lo), LD(hi), LD(a)
    l, h, w = X0 + A, X1 + A, LD(1.0 - nu)
    L = np.log1p((X1 - X0) / l)
    if nu == 1.0:
        e = np.expm1(R * L)
        xr, jr = X0 + l * e, l * (1 + e) * L
    elif nu < 1.0:
        rho = np.expm1(w * L)
        z = R * rho
        e = np.expm1(np.log1p(z) / w)
        xr, jr = X0 + l * e, l * (1 + e) * rho / (w * (1 + z))
    else:
        rho = np.expm1(-w * L)
        z = (1 - R) * rho
        xm = h * np.exp(np.log1p(z) / w)
        xr, jr = xm - A, -xm * rho / (w * (1 + z))
    # roundings: of the bounds and of the arguments of the exponentials, each up to |log| eps; the range
    # x_max - x_min enters relative to lo with the rounding of the shift by a
    tol = (24 + 8 * np.abs(L)) * EPS
    assert np.all(np.abs(LD(x) - xr) <= tol * np.maximum(xr, l))
    assert np.all((x >= lo) & (x <= hi))
    ok = hi > lo
    assert np.all(np.abs(LD(jac[ok]) - jr[ok]) <= (2 * tol * jr + 8 * EPS * (X0 + A))[ok])
    assert np.all(jac[~ok] == 0.0)


@pytest.mark.parametrize("jit", [False, True], ids=["interpreter", "compiled"])
def test_breit_wigner_map(torch_cuda, jit):
    rng = np.random.default_rng(9)
    n, M, G = 6000, 80.4, 2.1
    r = rng.random(n)
    r[:3] = 0.0, 1.0, 0.5
    lo = np.where(rng.random(n) < 0.4, 0.0, 10.0 ** rng.uniform(-6, 5, n))
    hi = lo + 10.0 ** rng.uniform(-6, 8, n)
    x, jac = run_op(torch_cuda, "INVARIANT_BW", [0, M, G, 1, 2], 2, [r, lo, hi], jit)
    mg, m2 = LD(M * G), LD(M * M)
    a, b = (LD(lo) - m2) / mg, (LD(hi) - m2) / mg
    D = np.arctan2((LD(hi) - LD(lo)) / mg, 1 + a * b)
    u = np.arctan(a) + D * LD(r)
    xr, jr = m2 + mg * np.tan(u), D * mg * (1 + np.tan(u) ** 2)
    # x moves by J/D per unit of angle, the angle carries a few roundings of pi
    scale = np.maximum(np.abs(xr), m2 * 0 + np.maximum(LD(lo), 0)) + jr / D * np.minimum(LD(1), np.abs(D))
    good = (r > 1e-6) & (r < 1 - 1e-6)  # at the ends the reference itself cancels
    assert np.all(np.abs(LD(x) - xr)[good] <= (32 * EPS * (scale + m2))[good])
    assert np.all((x >= lo) & (x <= hi)) and np.all(np.isfinite(jac)) and np.all(jac > 0)
