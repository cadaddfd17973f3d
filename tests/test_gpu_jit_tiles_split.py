"""Compiled mixed programs of more than six channels, which run several tiles a CTA when four or more CTAs of less than
256 threads are requested, against the same program with one tile a CTA: two and four tiles a CTA, one round of tiles
(spread over the CTAs, each group for itself) and several, empty channels, ragged and missing last tiles, with and
without VEGAS grids, generated, replayed and from explicit points.  The bars are those of test_gpu_jit_tiles.py, the
weights' for all but the near-threshold events (a last-bit difference moves them by FP32 roundings of a small
difference: one event in 10^3 up to 1e-3, and the cut decision of one in 10^4)."""
import numpy as np
import pytest

from paper_2602_06895_gb300 import ps
from paper_2602_06895_gb300 import workloads as W
from test_gpu_flow import torch_cuda  # noqa: F401

pytestmark = pytest.mark.gpu


def _close(a, b):
    n = a["weight"].size
    assert np.sum((a["weight"] == 0) != (b["weight"] == 0)) <= 1 + 1e-4 * n
    nz = (a["weight"] != 0) & (b["weight"] != 0)
    rel = np.abs(b["weight"][nz] / a["weight"][nz] - 1.0)
    assert rel.size == 0 or (np.median(rel) <= 5e-7 and np.sum(rel > 1e-3) <= 1 + 1e-3 * n)


@pytest.mark.parametrize("vegas", [False, True])
@pytest.mark.parametrize("counts", [[1, 0, 127, 128, 129, 1000, 65], [0, 0, 0, 0, 0, 0, 1], [40_001, 513, 0, 1, 0, 70, 900],
                                    [33_001] * 7])
def test_several_tiles_a_cta_match_one(torch_cuda, counts, vegas):  # noqa: F811
    torch = torch_cuda
    chans = W.channels_2to8()[:7]
    d = W.n_random_dims(chans[0])
    if vegas:
        chans = [dict(c, vegas_dims=d) for c in chans]
    n = sum(counts)
    res = []
    for block, ctas in ((128, 2), (128, 4), (64, 8)):
        prog = ps.program_for(chans, block_threads=block, ctas_per_sm=ctas, precision="mixed", jit=True)
        if vegas:
            for c in range(len(chans)):
                prog.set_vegas(c, W.vegas_grid_random(70 + c, d, 64))
        out, ws = prog.alloc(counts, 10, alpha=True)
        for v in out.values():
            v.fill_(-7.0)
        prog.generate(counts, 31, out, ws, event_offset=5)
        stats = prog.stats()
        replay, ws2 = prog.alloc(counts, 10, alpha=True)
        ex = prog.exec_create(counts, replay, ws2)
        ex.launch(31, 5)
        assert prog.stats() == stats
        for k in out:
            bits = [v[..., :n].contiguous().view(torch.int32) for v in (replay[k], out[k])]  # cut events may hold NaN
            assert torch.equal(*bits), k
            assert torch.all(out[k][..., n:] == -7.0), k  # nothing beyond the events
        w = out["weight"][:n].cpu().numpy()
        assert np.array_equal([s["n_nonzero"] for s in stats],
                              [np.count_nonzero(x) for x in np.split(w, np.cumsum(counts)[:-1])])
        point = torch.rand((d, 200), dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(3))
        pout, pws = prog.alloc([0, 200, 0, 0, 0, 0, 0], 10, alpha=True)
        prog.map(1, point, pout, pws)
        torch.cuda.synchronize()
        res.append(({"weight": w}, {"weight": pout["weight"][:200].cpu().numpy()}, stats))
    for k in (1, 2):
        _close(res[0][0], res[k][0])
        _close(res[0][1], res[k][1])
        for a, b in zip(res[0][2], res[k][2]):
            assert a["n"] == b["n"] and abs(b["sum_w"] - a["sum_w"]) <= 1e-4 * abs(a["sum_w"])
