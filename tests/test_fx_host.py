"""The integer/FP32 arithmetic of the FP64 update (su3_fx.cuh, su3_fx_kp.cuh) and its
tables, compiled for the host from the device's own header, against long double."""
import os
import re
import subprocess

import pytest

from paper_0904_1179_gb300 import build as su3_build

HERE = os.path.dirname(os.path.abspath(__file__))


def test_fx_arithmetic_on_host(tmp_path):
    exe = str(tmp_path / "fx_host")
    subprocess.run([su3_build.nvcc()] + su3_build.ARCH + ["-O2", "-std=c++17", "-I", su3_build.CSRC,
                                                          os.path.join(HERE, "fx_host.cu"), "-o", exe], check=True)
    out = subprocess.run([exe], capture_output=True, text=True)
    assert out.returncode == 0, out.stdout
    e = {k: float(v) for k, v in re.findall(r"(\w+) ([\d.]+)", out.stdout)}
    # units of 2^-53.  l has 24 bits of at most 2^31 units of 2^-62: 2^6 of them at most
    assert e["decode"] <= 0.13
    assert e["round_trip"] <= 0.63  # and half an ulp of the double
    # the largest error of a staple entry is below that of FP64 arithmetic with FMA on the same links
    assert e["staple"] < e["plain"], e
    # e0, d, e1 to about 2^-52.5 (the 24 FP32 roundings of sums up to 2^62 units of 2^-92), two of them on row 1
    assert e["reunitarise"] <= 4.0
    # ln 2 is 0.34 units of 2^-57 off, times up to 53 octaves, and a few roundings to 2^-57
    assert e["log"] <= 1.5
    # a sum of two products and its remainder in 24 bits: three roundings of at most 2^-54, and the table's
    assert e["trig"] <= 2.0
    assert e["root"] <= 2.0
    # root mean squares: no larger than in FP64
    assert e["dir"] <= e["dir_fp"] and e["azero"] <= e["azero_fp"] and e["avec"] <= e["avec_fp"], e
    # |R|^2 - 1: eight numbers of at most a few 2^-53 each
    assert e["unit"] <= 16.0
    assert e["flips"] == 0


def test_tables_are_correctly_rounded():
    mpmath = pytest.importorskip("mpmath")
    mpmath.mp.dps = 40
    text = open(os.path.join(su3_build.CSRC, "su3_fx_tables.cuh")).read()
    logs, trig = text.split("#define SU3_FX_TRIG_TABLE_PAIRS")
    logs = [int(v) for v in re.findall(r"(-?\d+)LL", logs)]
    trig = [int(v) for v in re.findall(r"(-?\d+)LL", trig)]
    assert len(logs) == 1025 and len(trig) == 2 * 513
    two = mpmath.mpf(2)
    for i, v in enumerate(logs):
        assert abs(mpmath.log(mpmath.mpf(1024 + i) / 2048) * two ** 57 - v) <= 0.5
    for j in range(513):
        x = 2 * mpmath.pi * j / 4096
        assert abs(mpmath.cos(x) * two ** 62 - trig[2 * j]) <= 0.5
        assert abs(mpmath.sin(x) * two ** 62 - trig[2 * j + 1]) <= 0.5
