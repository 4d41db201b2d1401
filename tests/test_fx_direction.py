"""The direction of a projected staple (fx_direction) where its length is a power of two: on the host against long
double, and on the GPU on configurations of the links 1 and diag(-1, -1, 1), whose projections are whole numbers."""
import os
import re
import subprocess

import numpy as np
import pytest

import oracle
from paper_0904_1179_gb300 import build as su3_build

HERE = os.path.dirname(os.path.abspath(__file__))


def test_directions_next_to_powers_of_two(tmp_path):
    exe = str(tmp_path / "fx_direction_host")
    subprocess.run([su3_build.nvcc()] + su3_build.ARCH + ["-O2", "-std=c++17", "-I", su3_build.CSRC,
                                                          os.path.join(HERE, "fx_direction_host.cu"), "-o", exe], check=True)
    out = subprocess.run([exe], capture_output=True, text=True)
    assert out.returncode == 0, out.stdout
    e = {k: float(v) for k, v in re.findall(r"(\w+) ([\d.]+)", out.stdout)}
    # components to 2^-56 and their squares' sum to about 2^-54 of itself; its root's reciprocal and the product add
    # two roundings of that size: four units of 2^-53
    assert e["direction"] <= 4.0
    assert e["length"] <= 4.0


def signed_identities(L, seed):
    """Links 1, a fifth of them diag(-1, -1, 1)."""
    u = oracle.cold_start(L)
    flip = np.random.default_rng(seed).random(u.shape[:5]) < 0.2
    u[flip, 0, 0, 0] = u[flip, 1, 1, 0] = -1.0
    return u


@pytest.mark.gpu
@pytest.mark.parametrize("lanes,decomp", [(1, None), (4, None), (0, None), (0, (2, 2, 1))])
def test_links_of_signed_identities(lanes, decomp):
    import paper_0904_1179_gb300 as su3
    L = (8, 4, 6, 4)
    given = signed_identities(L, 5)
    for mu in range(4):
        for parity in range(2):
            want = given.copy()
            oracle.half_sweep(L, 5.7, 3, 0, mu, parity, want)
            with su3.Lattice(L, 5.7, 3, start=su3.SU3_COLD, decomp=decomp) as lat:
                if lanes:
                    lat.set_lanes(lanes)
                lat.set_links(given)
                lat.half_sweep(mu, parity)
                got = lat.get_links()
            assert np.abs(got - want).max() <= 1e-12  # the bound of the parity tests
