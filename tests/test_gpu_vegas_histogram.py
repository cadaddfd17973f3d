"""The VEGAS training histogram over what it is given: odd and even numbers of mapped dimensions, event counts below and
above its 112 chunks, Philox and explicit points (64 bins: the number that every grid of the library has).  The reference
adds w^2 in extended precision: the kernel's sums carry at most one rounding per event of a bin."""
import numpy as np
import pytest

from paper_2602_06895_gb300 import ps
from paper_2602_06895_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch_cuda():
    import torch

    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2602_06895_gb300 import build

    build.build()
    return torch


@pytest.mark.parametrize("n", [1, 127, 5000, 100_003])
@pytest.mark.parametrize("dims", [1, 7, 8])
@pytest.mark.parametrize("explicit", [False, True], ids=["philox", "points"])
def test_histogram_sums(torch_cuda, n, dims, explicit):
    torch = torch_cuda
    ch = W.ww_hadronic(vegas_dims=dims)
    prog = ps.program_for([ch])
    bins = 64
    prog.vegas_training(True)
    out, ws = prog.alloc([n], 6)
    r = torch.tensor(W.uniform_r(3, n, 10).T.copy(), device="cuda")
    if explicit:
        prog.map(0, r, out, ws)
    else:
        import oracle as O

        prog.generate([n], 17, out, ws, event_offset=3)
        r = torch.tensor(O.random(17, 0, 3, n, 10).T.copy())
    h = prog.vegas_histogram(0, dims)
    w2 = out["weight"][:n].cpu().numpy().astype(np.longdouble) ** 2
    r = r.cpu().numpy()
    for j in range(dims):
        k = np.minimum((r[j] * bins).astype(int), bins - 1)
        ref, cnt = np.zeros(bins, np.longdouble), np.bincount(k, minlength=bins)
        np.add.at(ref, k, w2)
        assert np.all(np.abs(h[j] - ref) <= (cnt + 130) * 2.0 ** -53 * ref + 1e-300)


def test_a_new_seed_of_an_executor_reaches_the_histogram(torch_cuda):
    torch = torch_cuda
    chans = [dict(c, vegas_dims=5) for c in W.multichannel_2to5()]
    counts = [300, 0, 2000, 1, 129, 5000]
    res = []
    for replay in (False, True):
        prog = ps.program_for(chans)
        prog.vegas_training(True)
        out, ws = prog.alloc(counts, 7, alpha=True)
        if replay:
            ex = prog.exec_create(counts, out, ws)
            ex.launch(5, 10)
        else:
            prog.generate(counts, 5, out, ws, event_offset=10)
        torch.cuda.synchronize()
        res.append([prog.vegas_histogram(c, 5) for c in range(6)])
    for a, b in zip(*res):
        assert np.array_equal(a, b)
