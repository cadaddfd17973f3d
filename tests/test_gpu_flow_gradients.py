"""The training gradients at the edges of the backward GEMMs' 128-event tiles: batches of one event, of one
tile less or more an event, and hidden widths on and off the 128-column tile (16 takes the general GEMM and its own
column sums).  Only the last events carry weight, so that the rows of the last, ragged tile are the whole
gradient and a lost or doubled row shows in full.

Tolerance: the GEMM operands and adjoints are bfloat16 (2^-9 relative each, three products deep) and an
activation within FP32 rounding of a bfloat16 boundary may round the other way (2^-8 of one of the activations); with one
to five events carrying the gradient nothing averages out, so a parameter tensor may be off by a few times 2^-8:
5e-2 relative in the 2-norm."""
import numpy as np
import pytest

from paper_2602_06895_gb300 import ps
from test_gpu_flow import random_params, sample, torch_cuda  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("hidden,B", [(128, 1), (128, 127), (128, 129), (16, 130), (48, 257), (144, 1025)])
def test_last_events_gradients(torch_cuda, hidden, B):  # noqa: F811
    torch = torch_cuda
    fl = ps.Flow(5, 4, 8, hidden, max_batch=2048)
    p, orc, layout = random_params(fl, 23)
    fl.set_params(p)
    r, ld, _ = sample(torch, fl, B, 57)
    x = r.T
    w_map = (1.0 + x[:, 0] * x[:, 1] + x[:, 3]).contiguous()
    w_map[: max(0, B - 5)] = 0.0
    loss, g = fl.gradients(w_map)
    loss_o, grads_o = orc.loss_and_grads(x.cpu(), (w_map * torch.exp(ld)).cpu(), bf=True)
    assert abs(loss - loss_o) <= 1e-3 * max(1.0, abs(loss_o)), (loss, loss_o)
    for l, lay in enumerate(layout):
        for name, (o, _shape) in lay.items():
            ref = grads_o[l][name].numpy().ravel()
            got = g[o:o + ref.size].astype(np.float64)
            assert np.linalg.norm(got - ref) <= 5e-2 * np.linalg.norm(ref), (l, name)
