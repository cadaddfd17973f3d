"""Writes fp64_tables.h: the tables of the FP64 elementary functions of fp64_fast.cuh and of the
azimuth (map_device.cuh).  The values are computed at 60 significant digits with mpmath and rounded
to double; run once, the output is committed:

    python paper_2602_06895_gb300/csrc/gen_fp64_tables.py
"""
import os
import struct

import mpmath as mp

EXP_N, LOG_N, ATAN_N, TRIG_N = 256, 256, 64, 256


def split(v):
    """v as the nearest double and the nearest double of the rest."""
    hi = float(v)
    return hi, float(v - mp.mpf(hi))


def head(v, ulp):
    """v as its nearest multiple of ulp and the nearest double of the rest."""
    hi = float(mp.nint(v / ulp) * ulp)
    return hi, float(v - mp.mpf(hi))


def single(v):
    return struct.unpack("f", struct.pack("f", float(v)))[0]


def render():
    """The text of fp64_tables.h."""
    mp.mp.dps = 60
    ln2 = mp.log(2)
    exp2 = [split(mp.mpf(2) ** (mp.mpf(k) / EXP_N)) for k in range(EXP_N)]
    eh, el = head(ln2 / EXP_N, mp.mpf(2) ** -42)   # 34 bits: k eh is exact for |k| < 2^18
    lh, ll = head(ln2, mp.mpf(2) ** -41)
    inv, log = [], []
    for k in range(LOG_N + 1):
        c = single(mp.mpf(1) / (1 + mp.mpf(k) / LOG_N))
        inv.append(c)
        log.append(head(-mp.log(mp.mpf(c)), mp.mpf(2) ** -41))
    at = []
    for q in range(4):
        for k in range(ATAN_N + 1):
            a = mp.atan(mp.mpf(k) / ATAN_N)
            at.append(split((a, mp.pi / 2 - a, mp.pi / 2 + a, mp.pi - a)[q]))
    trig = []
    for k in range(TRIG_N):
        # the axes are exact: cos and sin of a multiple of pi/2 are not left to the rounding of pi
        c = {0: 1, TRIG_N // 4: 0, TRIG_N // 2: -1, 3 * TRIG_N // 4: 0}.get(k, mp.cos(2 * mp.pi * k / TRIG_N))
        s = {0: 0, TRIG_N // 4: 1, TRIG_N // 2: 0, 3 * TRIG_N // 4: -1}.get(k, mp.sin(2 * mp.pi * k / TRIG_N))
        trig.append((float(c), float(s)))

    def pairs(name, v):
        flat = [x for p in v for x in p]
        body = ",\n    ".join(", ".join(x.hex() for x in flat[i:i + 4]) for i in range(0, len(flat), 4))
        return f"static __device__ __align__(16) double {name}[{len(flat)}] = {{\n    {body}}};\n"

    def floats(name, v):
        body = ",\n    ".join(", ".join(x.hex() + "f" for x in v[i:i + 6]) for i in range(0, len(v), 6))
        return f"static __device__ float {name}[{len(v)}] = {{\n    {body}}};\n"

    return "\n".join([
        "// fp64_tables.h -- written by gen_fp64_tables.py (mpmath, 60 digits); do not edit.",
        "// Pairs (hi, lo) with hi + lo the value: kExpTab[k] = 2^(k/256); kLogTab[k] = -log(kLogInv[k]), hi a",
        "// multiple of 2^-41, kLogInv[k] the float nearest 256/(256 + k); kAtanTab[65 q + k] = atan(k/64),",
        "// pi/2 - atan, pi/2 + atan, pi - atan for q = 0..3; kTrigTab[k] = cos and sin of 2 pi k/256.",
        "// kExpStepHi + kExpStepLo = ln 2/256 and kLn2Hi + kLn2Lo = ln 2 with short heads.",
        "// The arrays are read-only global memory read through the read-only cache: indexed per thread,",
        "// they would serialise in the constant bank.",
        "#pragma once", "",
        f"constexpr double kExpStepHi = {eh.hex()}, kExpStepLo = {el.hex()};",
        f"constexpr double kLn2Hi = {lh.hex()}, kLn2Lo = {ll.hex()};",
        pairs("kExpTab", exp2), floats("kLogInv", inv), pairs("kLogTab", log), pairs("kAtanTab", at),
        pairs("kTrigTab", trig)])


def main():
    path = os.path.join(os.path.dirname(os.path.abspath(__file__)), "fp64_tables.h")
    with open(path, "w") as f:
        f.write(render())


if __name__ == "__main__":
    main()
