"""The sign of a zero quotient: a zero dividend of either sign over divisors of either sign, interpreted and compiled."""
import numpy as np
import pytest

from test_gpu_fp64_ops import run_op, torch_cuda  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("jit", [False, True], ids=["interpreter", "compiled"])
def test_zero_quotients_keep_their_sign(torch_cuda, jit):  # noqa: F811
    a, b = (x.ravel().copy() for x in np.meshgrid([0.0, -0.0], [1.0, -1.0, 3.0, -7.5e200, 1e-200, np.inf, -np.inf, 5e-324]))
    q, _ = run_op(torch_cuda, "DIV", [0, 1], 1, [a, b], jit)
    want = a / b
    assert np.array_equal(q, want) and np.array_equal(np.signbit(q), np.signbit(want))
