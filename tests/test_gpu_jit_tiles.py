"""Compiled mixed programs that run two tiles a CTA (several channels, four CTAs requested) against the same
program with one tile a CTA (two CTAs or none requested), through generate, explicit inputs and a captured replay: tiles
whose CTA spans two channels, empty channels, ragged and missing last tiles, with and without VEGAS grids (each
group of a CTA stages its channel's own).

Bars: both run the same device functions on the same Philox points; a different contraction of a product with a sum
can move one FP32 rounding, a few float ulps of a result: 5e-7 of a weight, and of a momentum component 5e-7 of the
event's energy scale.  Counts and cut decisions are equal, the sums of weights agree to 1e-6."""
import numpy as np
import pytest

from paper_2602_06895_gb300 import ps
from paper_2602_06895_gb300 import workloads as W
from test_gpu_flow import torch_cuda  # noqa: F401

pytestmark = pytest.mark.gpu


def _close(a, b):
    assert np.array_equal(a["weight"] == 0, b["weight"] == 0)
    nz = a["weight"] != 0
    assert np.all(np.abs(b["weight"][nz] / a["weight"][nz] - 1.0) <= 5e-7)
    for k in ("momenta", "x1", "x2", "alpha"):
        scale = np.max(np.abs(a[k]), axis=0) if a[k].ndim == 2 else 1.0
        assert np.all(np.abs(b[k] - a[k]) <= 5e-7 * scale), k


@pytest.mark.parametrize("vegas", [False, True])
@pytest.mark.parametrize("counts", [[1, 0, 127, 128, 129, 1000], [0, 0, 0, 0, 0, 1], [513, 1, 0, 40_001, 0, 0],
                                    [30_000] * 6])
def test_two_tiles_a_cta_match_one(torch_cuda, counts, vegas):  # noqa: F811
    torch = torch_cuda
    chans = W.multichannel_2to5()
    d = W.n_random_dims(chans[0])
    if vegas:
        chans = [dict(c, vegas_dims=d) for c in chans]
    res = []
    for ctas in (2, 4, 0):
        prog = ps.program_for(chans, ctas_per_sm=ctas, precision="mixed", jit=True)
        if vegas:
            for c in range(len(chans)):
                prog.set_vegas(c, W.vegas_grid_random(70 + c, d, 64))
        out, ws = prog.alloc(counts, 7, alpha=True)
        prog.generate(counts, 31, out, ws, event_offset=5)
        stats = prog.stats()
        torch.cuda.synchronize()
        host = {k: v.cpu().numpy() for k, v in out.items()}
        replay, ws2 = prog.alloc(counts, 7, alpha=True)
        ex = prog.exec_create(counts, replay, ws2)
        ex.launch(31, 5)
        assert prog.stats() == stats
        for k in out:
            assert torch.equal(replay[k], out[k]), k
        point = torch.rand((d, 200), dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(3))
        pout, pws = prog.alloc([0, 200, 0, 0, 0, 0], 7, alpha=True)
        prog.map(1, point, pout, pws)
        torch.cuda.synchronize()
        res.append((host, stats, {k: v.cpu().numpy() for k, v in pout.items()}))
    n = sum(counts)
    out = [{k: v[..., :n] for k, v in r[0].items()} for r in res]
    for k in (1, 2):
        _close(out[0], out[k])
        _close(res[0][2], res[k][2])
        for a, b in zip(res[0][1], res[k][1]):
            assert a["n"] == b["n"] and a["n_nonzero"] == b["n_nonzero"]
            assert abs(b["sum_w"] - a["sum_w"]) <= 1e-6 * abs(a["sum_w"])
