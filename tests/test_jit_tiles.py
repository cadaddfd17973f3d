"""Which compiled mixed programs run several tiles a CTA (host only, from the generated kernel's launch bounds)."""
import ctypes as C

import pytest

from paper_2602_06895_gb300 import ps
from paper_2602_06895_gb300 import workloads as W


@pytest.mark.parametrize("chans, block, ctas, bounds", [
    (W.multichannel_2to5(), 128, 4, "128, 4"),      # six channels in one unit: one tile a CTA
    (W.channels_2to8()[:7], 128, 4, "256, 2"),      # one unit a channel: 256 threads
    (W.channels_2to8()[:7], 64, 8, "256, 2"),
    (W.channels_2to8()[:7], 128, 0, "256, 2")], ids=lambda v: str(len(v)) if isinstance(v, list) else str(v))
def test_tiles_of_a_mixed_program(monkeypatch, tmp_path, chans, block, ctas, bounds):
    dump = tmp_path / "src.cu"
    monkeypatch.setenv("PS_JIT_DUMP", str(dump))
    graphs = [ps.build_channel(chans, c) for c in range(len(chans))]
    hs = (C.c_void_p * len(chans))(*[g.h.value for g in graphs])
    opt = ps.Options(block, ctas, ps.PRECISION["mixed"], ps.PS_PROGRAM_JIT)
    log = C.create_string_buffer(1 << 16)
    assert ps.lib().ps_jit_check(hs, len(chans), C.byref(opt), log, len(log)) == 0, log.value
    assert f"__launch_bounds__({bounds})" in dump.read_text()
