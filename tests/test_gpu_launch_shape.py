"""The launch shapes that the library picks by itself -- blocks of one warp for FP32 half-sweeps under 0.8 waves, tiles of
64 or 32 for the automatic schedule where an x3 layer is no whole number of 128 -- against eight launches of 128 threads:
the same links and acceptance counts, bit for bit."""
import numpy as np
import pytest

import paper_0904_1179_gb300 as su3

pytestmark = pytest.mark.gpu

PHASES, PER_DIRECTION, CHAINED = su3.SU3_SCHED_PHASES, su3.SU3_SCHED_PER_DIRECTION, su3.SU3_SCHED_CHAINED


# waves and tiles on a GPU of 152 SMs
@pytest.mark.parametrize("dims,precision,schedule", [
    ((20, 20, 20, 20), su3.SU3_FP64, PER_DIRECTION),       # 1.4 waves, tiles of 32
    ((20, 20, 24, 20), su3.SU3_FP64, PER_DIRECTION),       # 1.6, 64
    ((22, 22, 22, 20), su3.SU3_FP64, PHASES),              # no whole tiles
    ((26, 24, 24, 24), su3.SU3_FP32_MIXED, CHAINED),       # 1.2, 64
    ((28, 28, 28, 28), su3.SU3_FP32_EFT, CHAINED),         # 2.0, 32
    ((36, 36, 36, 36), su3.SU3_FP32_MIXED, PHASES),        # tiles of 32 only, over three waves
    ((14, 6, 10, 14), su3.SU3_FP32_MIXED, PHASES),         # single-site store, a twentieth of a wave
    ((18, 10, 14, 22), su3.SU3_FP32_EFT, PHASES),
    ((16, 14, 14, 16), su3.SU3_FP32_MIXED, PHASES),        # one thread per link of the site-paired store
    ((20, 18, 18, 20), su3.SU3_FP32_MIXED, PHASES),        # one thread per pair
    ((22, 22, 22, 24), su3.SU3_FP32_EFT, PHASES),           # 0.75 waves
    ((24, 24, 24, 20), su3.SU3_FP32_MIXED, PHASES),        # 0.9: blocks of 128
])
@pytest.mark.parametrize("tries", [1, 8])
def test_automatic_launch_shapes_give_the_same_bits(dims, precision, schedule, tries):
    with su3.Lattice(dims, 5.7, 17, start=su3.SU3_HOT, precision=precision) as a, \
         su3.Lattice(dims, 5.7, 17, start=su3.SU3_HOT, precision=precision) as b:
        b.set_block_size(128)
        b.set_schedule(PHASES)
        assert a.schedule == schedule
        for lat in (a, b):
            lat.set_heatbath(tries)
            lat.set_stats(True)
            lat.sweep(2)
            lat.half_sweep(1, 1)
        assert a.stats() == b.stats()
        assert np.array_equal(a.get_links(), b.get_links())


def test_set_block_size_keeps_its_tiles():
    with su3.Lattice((20, 20, 20, 20), 5.7, 1, precision=su3.SU3_FP64) as lat:
        with pytest.raises(su3.Su3Error):
            lat.set_schedule(PER_DIRECTION)  # the default block of 128 does not divide a layer
        assert lat.schedule == PER_DIRECTION
        lat.set_block_size(128)
        assert lat.schedule == PHASES
        lat.set_block_size(32)
        assert lat.schedule == PER_DIRECTION
        lat.set_block_size(64)
        assert lat.schedule == PHASES
        lat.set_block_size(0)
        assert lat.schedule == PER_DIRECTION
