"""An interpreted program whose CTA fills the shared memory to the last word still is a program when the library would
add a constant of its own to it (the logarithm of a power-law map between constant bounds).  The map of the full
program is that of a small one, to the rounding of that logarithm (24 + 8 |L| roundings, as in test_gpu_fp64_ops.py)."""
import numpy as np
import pytest

from paper_2602_06895_gb300 import ps
from test_gpu_flow import torch_cuda  # noqa: F401

pytestmark = pytest.mark.gpu

EPS = 2.0 ** -52
INPUTS, LIVE = 60, 104  # scalars live to the end: 256 x 8 bytes of shared memory each


def _graph(xmin, squares, adds, inputs=INPUTS, live=LIVE):
    """The map of r0 between xmin and 5 (nu = 0.3, no mass), `squares` (20 bytes of code) and `adds` (24 bytes) on the
    second input, and a sum over all inputs and their like."""
    g = ps.Graph.create(inputs)
    x, j = g.add("INVARIANT_NU", [0, 0.0, 0.3, xmin, 5.0, 0.0], 2)
    v = 1
    for _ in range(squares):
        v = g.add("SQUARE", [v], 1)[0]
    for _ in range(adds):
        v = g.add("ADD", [v, 0.0], 1)[0]
    kept = list(range(1, inputs)) + [g.add("SQUARE", [1], 1)[0] for _ in range(live - inputs)]
    for k in kept:
        v = g.add("ADD", [v, k], 1)[0]
    g.set_outputs([x, j, v], [ps.ROLE_X1, ps.ROLE_X2, ps.ROLE_WEIGHT])
    return g


def _program(*args):
    try:
        return ps.Program([_graph(*args)], block_threads=256)
    except ps.PSError:
        return None


def test_a_full_cta_keeps_its_program(torch_cuda):  # noqa: F811
    torch = torch_cuda
    # without a derived constant (x_min = a = 0 leaves the map without a range): fill up to the last four bytes
    lo, hi = 0, 2000
    assert _program(0.0, lo, 0) is not None and _program(0.0, hi, 0) is None
    while hi - lo > 1:
        mid = (lo + hi) // 2
        lo, hi = (mid, hi) if _program(0.0, mid, 0) is not None else (lo, mid)
    adds = 0
    while lo > 0 and _program(0.0, lo - 1, adds + 1) is not None:
        lo, adds = lo - 1, adds + 1
    # as many words of code and immediates, and now a range between constants
    full = _program(0.3, lo, adds)
    assert full is not None
    small = _program(0.3, 0, 0, 2, 2)
    r = np.random.default_rng(2).random((INPUTS, 3000))
    res = []
    for prog, rows in ((full, INPUTS), (small, 2)):
        out, ws = prog.alloc([3000], 0)
        prog.map(0, torch.tensor(r[:rows].copy(), device="cuda"), out, ws)
        res.append([out[k].cpu().numpy() for k in ("x1", "x2")])
    tol = (24 + 8 * np.log1p((5.0 - 0.3) / 0.3)) * EPS
    for a, b in zip(*res):
        assert np.all(np.abs(a - b) <= tol * np.abs(b))
