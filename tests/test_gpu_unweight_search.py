"""The search for the maximum weight beyond what the short lists of the other tests reach: a sampled first guess
(2^20 weights and more) that is right, too high (the tail hides from the sample) or too long for the tail
list, ties, subnormal and huge weights; and the selection's FP32 bounds against FP64 at extreme scales."""
import numpy as np
import pytest

from oracle import unweight as U
from paper_2602_06895_gb300 import ps

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch_cuda():
    import torch

    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2602_06895_gb300 import build

    build.build()
    return torch


N = (1 << 20) + 4099


def _weights(kind):
    g = np.random.default_rng(11)
    w = g.lognormal(0.0, 0.4, N)
    if kind == "hidden_tail":  # a few large weights where the sample does not look
        w[:] = 1.0
        w[256 * 7 + 3] = 400.0
    elif kind == "sampled_tail":  # large weights only where it does
        w[:] = 1.0
        w[:64] = 30.0
    elif kind == "ties":
        w = np.where(g.random(N) < 0.3, 2.5, 1.0)
    elif kind == "subnormal":
        w = w * 1e-310
    elif kind == "huge":
        w = w * 1e300
    elif kind == "few":
        w = w * (g.random(N) < 1e-4)
    return w


@pytest.mark.parametrize("kind", ["smooth", "hidden_tail", "sampled_tail", "ties", "subnormal", "huge", "few"])
@pytest.mark.parametrize("eps", [1e-4, 1e-2, 0.6])
def test_search_and_selection(torch_cuda, kind, eps):
    torch = torch_cuda
    w = _weights(kind)
    uw = ps.Unweighter(N)
    wd = torch.tensor(w, device="cuda")
    uw.max_weight(wd, eps)
    idx = torch.empty(N, dtype=torch.int64, device="cuda")
    wo = torch.empty(N, dtype=torch.float64, device="cuda")
    uw.select(wd, 3, idx, wo, event_offset=5)
    torch.cuda.synchronize()
    t, S, m, above, bad = uw.result.tolist()
    # the root is (A - eps S)/K with S and A sums of up to 2^20 terms: their roundings, 2^10 eps at most
    assert t == pytest.approx(U.max_weight(w, eps), rel=1e-12, abs=1e-320)
    assert m == w.max() and bad == 0
    assert above == np.count_nonzero(w > t)
    na = int(uw.n_accepted.item())
    i_o, w_o = U.accept(w, t, seed=3, ev0=5)
    assert np.array_equal(idx[:na].cpu().numpy(), i_o)
    assert np.array_equal(wo[:na].cpu().numpy(), w_o)
