"""Programs compiled one unit per channel build at every CTA size and count that one unit of all channels takes: the
channel units keep to the registers that the CTAs leave a thread, also above 256 threads without a requested count and
where an SM's warps are no multiple of four.  Host only (NVRTC and nvJitLink)."""
import ctypes as C

import pytest

from paper_2602_06895_gb300 import ps
from paper_2602_06895_gb300 import workloads as W

SETS = {"2to5x3": W.multichannel_2to5()[:3], "2to5x6": W.multichannel_2to5(), "2to8x3": W.channels_2to8()[:3],
        "2to8x6": W.channels_2to8()[:6], "2to8x7": W.channels_2to8()[:7]}
CASES = [(name, "f64", block, ctas) for name in ("2to5x3", "2to8x3")
         for block, ctas in ((288, 0), (384, 0), (416, 0), (512, 0), (320, 1), (160, 2))]
CASES += [("2to5x6", "f64", 512, 0), ("2to8x6", "f64", 320, 0), ("2to8x6", "f64", 512, 0)]
CASES += [("2to8x7", "mixed", block, ctas) for block, ctas in ((96, 0), (224, 0), (64, 5))]


@pytest.mark.parametrize("name, precision, block, ctas", CASES)
def test_split_program_builds(name, precision, block, ctas):
    chans = SETS[name]
    graphs = [ps.build_channel(chans, c) for c in range(len(chans))]
    hs = (C.c_void_p * len(chans))(*[g.h.value for g in graphs])
    opt = ps.Options(block, ctas, ps.PRECISION[precision], ps.PS_PROGRAM_JIT)
    log = C.create_string_buffer(1 << 16)
    assert ps.lib().ps_jit_check(hs, len(chans), C.byref(opt), log, len(log)) == 0, log.value


def test_register_cap_of_a_block(monkeypatch, tmp_path):
    """65536 registers in four banks that the warps share in turn: 11 warps (352 threads) put three in a bank,
    16384 / 96 = 170, in steps of 8; the cap of 168 that suits small CTAs gives way to 128 at 512 threads."""
    dump = tmp_path / "src.cu"
    monkeypatch.setenv("PS_JIT_DUMP", str(dump))
    for name, block, cap in (("2to8x3", 352, 168), ("2to5x3", 512, 128), ("2to5x3", 128, 168)):
        ps.jit_check(SETS[name], block, "f64")
        assert dump.read_text().rstrip().endswith(f"// maxrregcount {cap}")
