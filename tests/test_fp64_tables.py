"""The tables of the FP64 elementary functions (csrc/fp64_tables.h) are the output of their generator, and
their pairs carry the values to about 100 bits."""
import importlib.util
import os
import re

import pytest

mp = pytest.importorskip("mpmath")

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2602_06895_gb300", "csrc")


def test_header_is_the_generators_output_and_accurate():
    spec = importlib.util.spec_from_file_location("gen_fp64_tables", os.path.join(CSRC, "gen_fp64_tables.py"))
    gen = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(gen)
    text = open(os.path.join(CSRC, "fp64_tables.h")).read()
    assert text == gen.render()
    mp.mp.dps = 50
    arr = {n: [float.fromhex(v.strip().rstrip("f")) if "p" in v else float(v) for v in body.split(",") if v.strip()]
           for n, body in re.findall(r"(k\w+)\[\d+\] = \{([^}]*)\}", text)}
    for k in range(256):
        hi, lo = arr["kExpTab"][2 * k:2 * k + 2]
        assert abs((mp.mpf(hi) + mp.mpf(lo)) / mp.mpf(2) ** (mp.mpf(k) / 256) - 1) < mp.mpf(2) ** -100
        c, s = arr["kTrigTab"][2 * k:2 * k + 2]
        assert abs(c - mp.cos(mp.pi * k / 128)) < 2.0 ** -53 and abs(s - mp.sin(mp.pi * k / 128)) < 2.0 ** -53
    for k in range(257):
        hi, lo = arr["kLogTab"][2 * k:2 * k + 2]
        assert abs(mp.mpf(hi) + mp.mpf(lo) + mp.log(mp.mpf(arr["kLogInv"][k]))) < mp.mpf(2) ** -90
    for q, sign in enumerate((1, -1, 1, -1)):
        for k in range(65):
            hi, lo = arr["kAtanTab"][2 * (65 * q + k):2 * (65 * q + k) + 2]
            v = (0, mp.pi / 2, mp.pi / 2, mp.pi)[q] + sign * mp.atan(mp.mpf(k) / 64)
            assert abs(mp.mpf(hi) + mp.mpf(lo) - v) < mp.mpf(2) ** -100
