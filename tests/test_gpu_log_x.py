"""log x1 and log x2 of r_to_x1x2 as results of their own: (r, 1 - r) log(s / S) to a few roundings, also where one of
them is a small part of the other, and as the argument of a single density; the pair of densities of the library's own
channels gives the same value from them to the roundings of log x2.

Bounds: s/S carries two roundings, 2 eps absolute in its logarithm L, the logarithm two more, each result one: (4 + 2/|L|)
eps relative to the result, doubled."""
import numpy as np
import pytest

from paper_2602_06895_gb300 import ps
from test_gpu_fp64_ops import EPS, LD, torch_cuda  # noqa: F401

pytestmark = pytest.mark.gpu

S, AL, BE = 169.0e6, -1.1, 3.0


def _run(torch, outputs, cols, jit):
    """r_to_x1x2 with the logarithms on (r, s), then outputs(g, x1, x2, l1, l2) -> (a, b)."""
    g = ps.Graph.create(2)
    x1, x2, _, l1, l2 = g.add("R_TO_X1X2", [0, 1, S, 1.0], 5)
    a, b = outputs(g, x1, x2, l1, l2)
    g.set_outputs([a, b, a], [ps.ROLE_X1, ps.ROLE_X2, ps.ROLE_WEIGHT])
    prog = ps.Program([g], jit=jit)
    out, ws = prog.alloc([cols.shape[1]], 0)
    prog.map(0, torch.tensor(cols, device="cuda"), out, ws)
    return out["x1"].cpu().numpy(), out["x2"].cpu().numpy()


@pytest.mark.parametrize("jit", [False, True], ids=["interpreter", "compiled"])
def test_logarithms(torch_cuda, jit):  # noqa: F811
    rng = np.random.default_rng(19)
    n = 20000
    r = rng.random(n)
    r[: n // 4] = 1.0 - 10.0 ** rng.uniform(-12, -1, n // 4)
    r[n // 4: n // 2] = 10.0 ** rng.uniform(-12, -1, n // 4)
    s = S * np.exp(-rng.uniform(0.05, 25.0, n))
    cols = np.stack([r, s])
    l1, l2 = _run(torch_cuda, lambda g, x1, x2, a, b: (a, b), cols, jit)
    L = np.log(LD(s) / LD(S))
    tol = 2 * (4 + 2 / np.abs(L)) * EPS
    assert np.all(np.abs(LD(l1) - LD(r) * L) <= tol * np.abs(LD(r) * L))
    assert np.all(np.abs(LD(l2) - (1 - LD(r)) * L) <= tol * np.abs((1 - LD(r)) * L))
    # one density of x2 from its logarithm, and the pair
    one, both = _run(torch_cuda, lambda g, x1, x2, a, b: (g.add("PDF_POWER", [x2, AL, BE, b], 1)[0],
                                                          g.add("PDF_POWER", [x1, AL, BE, a, x2, b], 1)[0]), cols, jit)
    X1, X2 = (v.astype(LD) for v in _run(torch_cuda, lambda g, x1, x2, a, b: (x1, x2), cols, jit))
    ref = np.exp(LD(AL) * (1 - LD(r)) * L) * (1 - X2) ** 3
    pair = np.exp(LD(AL) * L) * (1 - X1) ** 3 * (1 - X2) ** 3
    wide = (16 + 8 * np.abs(L)) * EPS  # the exponent's absolute error, and the powers
    assert np.all(np.abs(LD(one) - ref) <= wide * ref)
    assert np.all(np.abs(LD(both) - pair) <= wide * pair)
