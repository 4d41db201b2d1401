"""The integer/FP32 arithmetic of the FP64 update (su3_fx.cuh), compiled for the
host from the device's own header, against long double."""
import os
import re
import subprocess

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
