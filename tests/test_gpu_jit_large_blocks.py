"""Compiled programs in CTAs above 256 threads and of an odd number of warps against the 128-thread form: the same device
functions on the same Philox points, so that only a different contraction of a product with a sum can move a rounding
(the bounds of the 512-thread test of test_gpu_jit.py; at 2->8, where an event near a threshold amplifies a
rounding, of its 2->8 test)."""
import numpy as np
import pytest

from paper_2602_06895_gb300 import ps
from paper_2602_06895_gb300 import workloads as W
from test_gpu_flow import torch_cuda  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("channels, precision, n_ch, block, ctas", [
    (W.multichannel_2to5, "f64", 3, 288, 0), (W.multichannel_2to5, "f64", 3, 512, 0), (W.multichannel_2to5, "f64", 6, 416, 0),
    (W.multichannel_2to5, "f64", 6, 320, 1), (W.multichannel_2to5, "f64", 3, 160, 2), (W.channels_2to8, "f64", 3, 288, 0),
    (W.channels_2to8, "f64", 6, 384, 0), (W.channels_2to8, "f64", 6, 512, 0), (W.channels_2to8, "mixed", 7, 96, 0),
    (W.channels_2to8, "mixed", 7, 224, 0)])
def test_cta_shapes_match_128_threads(torch_cuda, channels, precision, n_ch, block, ctas):  # noqa: F811
    chans = channels()[:n_ch]
    counts = [700, 30_001, 0, 25_000, 40_959, 513, 6000][:n_ch]
    res = []
    for b, k in ((128, 0), (block, ctas)):
        prog = ps.program_for(chans, block_threads=b, ctas_per_sm=k, precision=precision, jit=True)
        out, ws = prog.alloc(counts, chans[0]["n"] + 2, alpha=True)
        prog.generate(counts, 99, out, ws)
        res.append((prog.stats(), out["weight"].cpu().numpy()))
    (sa, wa), (sb, wb) = res
    nz = (wa != 0) & (wb != 0)
    rel = np.abs(wb[nz] / wa[nz] - 1.0)
    if channels is W.multichannel_2to5:
        assert np.array_equal(wa == 0, wb == 0) and rel.max() < 1e-12
        bound = 1e-13
    else:
        assert np.sum((wa == 0) != (wb == 0)) <= 1e-4 * wa.size
        assert np.median(rel) <= (1e-12 if precision == "f64" else 1e-3)
        bound = 1e-9 if precision == "f64" else 1e-4
    for a, b in zip(sa, sb):
        assert a["n"] == b["n"] and abs(b["sum_w"] - a["sum_w"]) <= bound * abs(a["sum_w"])
