"""The inverse map of records that hold no event: NaN momenta give NaN in every dimension taken from them, also where the
bounds of an invariant fall together for them, and leave the records beside them as they were."""
import numpy as np
import pytest

from paper_2602_06895_gb300 import ps
from paper_2602_06895_gb300 import workloads as W
from test_gpu_flow import torch_cuda  # noqa: F401

pytestmark = pytest.mark.gpu


def test_nan_momenta_give_nan(torch_cuda):  # noqa: F811
    torch = torch_cuda
    ch = W.multichannel_2to5()[4]  # s-channel invariants only, Breit-Wigner and power law
    ch = dict(ch, integrand="none")
    prog = ps.program_for([ch])
    n, d = 1000, W.n_random_dims(ch)
    out, ws = prog.alloc([n], 7)
    prog.generate([n], 4, out, ws)
    bad = torch.arange(n, device="cuda") % 7 == 3
    rows = []
    for mom in (out["momenta"][:, :n].contiguous(), torch.where(bad, torch.nan, out["momenta"][:, :n]).contiguous()):
        r = torch.empty((d, n), dtype=torch.float64, device="cuda")
        ps.inverse_map(prog, 0, ch, mom, out["x1"][:n].contiguous(), out["x2"][:n].contiguous(), r)
        rows.append(r.cpu().numpy())
    bad = bad.cpu().numpy()
    x_dims = [0, 1 + len(ch["sorder"])]  # s-hat and the x1, x2 split come from x1 and x2
    rest = [j for j in range(d) if j not in x_dims]
    assert np.all(np.isnan(rows[1][rest][:, bad]))
    assert np.array_equal(rows[1][:, ~bad], rows[0][:, ~bad]) and np.all(np.isfinite(rows[0]))
