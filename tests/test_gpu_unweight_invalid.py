"""Invalid weights among 2^20 and more: they are skipped and counted also where they hide the valid ones from the
sample (one weight in eight, the first 256 of each 2048 of a block's chunk) that says whether the tail fits its list.
A list that overflows is never searched: the root is the one of all valid weights, the same bit for bit each time."""
import numpy as np
import pytest

from oracle import unweight as U
from paper_2602_06895_gb300 import ps
from test_gpu_flow import torch_cuda  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1 << 22, 1_500_003])
@pytest.mark.parametrize("eps", [1e-3, 1e-2, 0.6])
@pytest.mark.parametrize("hidden", [1.0, 0.95])
def test_invalid_weights_at_the_sampled_positions(torch_cuda, n, eps, hidden):  # noqa: F811
    torch = torch_cuda
    g = np.random.default_rng(17)
    w = g.exponential(1.0, n)
    chunk = -(-n // 512)
    sampled = (np.arange(n) % chunk) % 2048 < 256
    bad = sampled & (g.random(n) < hidden)
    w[bad] = np.where(g.random(n) < 0.5, -1.0, np.nan)[bad]
    uw = ps.Unweighter(n)
    wd = torch.tensor(w, device="cuda")
    runs = []
    for _ in range(3):
        uw.max_weight(wd, eps)
        runs.append(uw.result.cpu().numpy().copy())
    valid = w[~bad]
    t, S, m, above, n_bad = runs[0]
    # sums of up to 2^22 terms in trees and exact limbs: far below 2^11 roundings
    assert t == pytest.approx(U.max_weight(valid, eps), rel=1e-12)
    assert S == pytest.approx(valid.sum(), rel=1e-12) and m == valid.max() and n_bad == bad.sum()
    assert above == np.count_nonzero(valid > t)
    assert all(np.array_equal(runs[0], r) for r in runs[1:])
