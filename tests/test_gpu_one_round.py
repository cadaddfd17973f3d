"""Interpreted launches whose tiles all fit on the device at once take a CTA per tile when no CTA count is
requested; a requested count keeps its own grid.  Tiles and the order of their sums do not depend on the grid, so
outputs and statistics are equal bit for bit, at the edges of the rule's range (four CTAs an SM, as many as fit),
through generate and a captured replay."""
import pytest

from paper_2602_06895_gb300 import ps
from paper_2602_06895_gb300 import workloads as W
from test_gpu_flow import torch_cuda  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["f64", "mixed"])
@pytest.mark.parametrize("per_sm,extra", [(4, 0), (4, 1), (5, -63), (8, 0), (8, 1), (16, 128)])
def test_one_round_matches_a_requested_grid(torch_cuda, precision, per_sm, extra):  # noqa: F811
    torch = torch_cuda
    n = [torch.cuda.get_device_properties(0).multi_processor_count * per_sm * 128 + extra]
    res = []
    for ctas in (0, 4):
        prog = ps.program_for([W.two_body_fixed()], ctas_per_sm=ctas, precision=precision)
        out, ws = prog.alloc(n, 4, x=False)
        prog.generate(n, 17, out, ws, event_offset=3)
        stats = prog.stats()
        replay, ws2 = prog.alloc(n, 4, x=False)
        prog.exec_create(n, replay, ws2).launch(17, 3)
        assert prog.stats() == stats
        torch.cuda.synchronize()
        assert all(torch.equal(out[k], replay[k]) for k in out)
        res.append((out, stats))
    assert res[0][1] == res[1][1]
    for k in res[0][0]:
        assert torch.equal(res[0][0][k], res[1][0][k]), k
