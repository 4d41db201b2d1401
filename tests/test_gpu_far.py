"""FP64 configurations with a link far from SU(3), which take the update in FP64 arithmetic: what that is limited to,
and every kernel that holds it."""
import contextlib

import numpy as np
import pytest

import oracle
import paper_0904_1179_gb300 as su3

pytestmark = pytest.mark.gpu

MIX = [(4, 4, 4, 4), (6, 4, 10, 8), (8, 8, 8, 8)]
BETAS = [5.7, 5.5, 6.0]
SEEDS = [11, 12, 13]


def with_far_link(L, seed, kind):
    u = oracle.hot_start(L, seed)
    if kind == "nan":
        u[0, 1, 1, 0, 2] = np.nan
    else:
        u[0, 1, 1, 0, 2] *= 1.5
    return u


@pytest.mark.parametrize("kind", ["stretched", "nan"])
@pytest.mark.parametrize("tries", [1, 4])
def test_replicas_of_a_batch_are_independent(kind, tries):
    # The far link of one replica changes no bit of another, which equals the lattice alone; its own replica equals
    # its lattice too.  A proper configuration, or a sweep, brings the replica back.
    far = with_far_link(MIX[1], 7, kind)
    with su3.Batch(MIX, BETAS, SEEDS, start=su3.SU3_HOT, precision=su3.SU3_FP64) as b, contextlib.ExitStack() as stack:
        alone = [stack.enter_context(su3.Lattice(L, BETAS[r], SEEDS[r], start=su3.SU3_HOT)) for r, L in enumerate(MIX)]
        b.set_heatbath(tries)
        for lat in alone:
            lat.set_heatbath(tries)
        b.set_links(1, far)
        alone[1].set_links(far)
        for step in range(3):
            if step == 2:
                proper = oracle.hot_start(MIX[1], 8)
                b.set_links(1, proper)
                alone[1].set_links(proper)
            plaq = b.plaquettes()
            for r, lat in enumerate(alone):
                assert np.array_equal(b.get_links(r), lat.get_links(), equal_nan=True), (step, r)
                assert np.array_equal(plaq[r], su3.load_library().su3_plaquette(lat.handle), equal_nan=True), (step, r)
            b.sweep(1)
            for lat in alone:
                lat.sweep(1)


PHASES = [(mu, parity) for mu in range(4) for parity in range(2)]


@pytest.mark.parametrize("L,decomp", [((8, 4, 6, 4), None), ((16, 16, 16, 16), None), ((8, 4, 8, 4), (2, 2, 1))])
def test_eight_half_sweeps_end_the_fp64_arithmetic(L, decomp):
    # A chain driven by half-sweeps is the chain of sweeps, bit for bit: once all eight have rewritten the far link
    # and its neighbours, it is back in the arithmetic of proper configurations.
    far = with_far_link(L, 3, "stretched")
    with su3.Lattice(L, 5.7, 5, decomp=decomp) as a, su3.Lattice(L, 5.7, 5, decomp=decomp) as b:
        a.set_links(far)
        b.set_links(far)
        for t in range(3):
            a.sweep(1)
            for mu, parity in PHASES:
                b.half_sweep(mu, parity)
            b.sweep_count = t + 1
            assert np.array_equal(a.get_links(), b.get_links()), t
            assert a.plaquette() == b.plaquette()


@pytest.mark.parametrize("decomp", [None, (2, 2, 1)])
def test_half_sweeps_around_a_sweep_do_not_end_it(decomp):
    # Four half-sweeps, a sweep, the other four: not all links were rewritten since the sweep found its NaN, which
    # stays the only one.
    L = (8, 4, 8, 4)
    ref = oracle.hot_start(L, 3)
    bad = with_far_link(L, 3, "nan")
    with su3.Lattice(L, 5.7, 5, decomp=decomp) as lat:
        lat.set_links(bad)
        for mu, parity in PHASES[:4]:
            lat.half_sweep(mu, parity)
        lat.sweep(1)
        for mu, parity in PHASES[4:] + PHASES:
            lat.half_sweep(mu, parity)
        u = lat.get_links()
    lost = np.isnan(u).any(axis=(-1, -2, -3))
    assert lost.sum() == 1 and lost[0, 1, 1, 0, 2]
    # the plaquettes of the lost link hold links whose staples were no numbers: they have never changed
    assert np.abs(u - ref)[0, 1, 1, 0, 0].max() <= 1e-12


@pytest.mark.parametrize("kind", ["stretched", "nan"])
@pytest.mark.parametrize("tries", [1, 4])
@pytest.mark.parametrize("L,threads", [((8, 8, 4, 4), 32), ((16, 16, 16, 8), 128)])
def test_every_kernel_holds_the_same_update(kind, tries, L, threads):
    # One thread per link in eight launches, against four and the automatic number of lanes, the per-direction and the
    # chained launches and the measuring sweep: the same links, bit for bit, and the plaquettes of each sweep.
    far = with_far_link(L, 6, kind)

    def lattice():
        lat = su3.Lattice(L, 5.7, 5)
        lat.set_heatbath(tries)
        lat.set_links(far)
        return lat

    with lattice() as lat:
        lat.set_lanes(1)
        lat.set_schedule(su3.SU3_SCHED_PHASES)
        plaquettes = []
        for _ in range(2):
            lat.sweep(1)
            plaquettes.append(su3.load_library().su3_plaquette(lat.handle))
        want = lat.get_links()
    for lanes, schedule in ((4, None), (0, None), (1, su3.SU3_SCHED_PER_DIRECTION), (1, su3.SU3_SCHED_CHAINED)):
        with lattice() as lat:
            lat.set_lanes(lanes)
            if schedule is not None:
                lat.set_block_size(threads)
                lat.set_schedule(schedule)
            lat.sweep(2)
            assert np.array_equal(lat.get_links(), want, equal_nan=True), (lanes, schedule)
    with lattice() as lat:
        measured = lat.sweep_measured(2)
        assert np.array_equal(lat.get_links(), want, equal_nan=True)
    np.testing.assert_allclose(measured, plaquettes, rtol=0, atol=1e-13)  # the bound of the parity tests
