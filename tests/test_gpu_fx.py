"""FP64 stores: the update on the integer and FP32 pipes (su3_fx.cuh) and the
configurations it leaves to FP64 arithmetic (links far from SU(3)), on the
GPU against the oracle and against each other.
"""
import numpy as np
import pytest

import oracle
import paper_0904_1179_gb300 as su3

pytestmark = pytest.mark.gpu

BETA = 5.7


def half_sweep(L, links, mu, parity, lanes=0, decomp=None, seed=3):
    with su3.Lattice(L, BETA, seed, start=su3.SU3_COLD, decomp=decomp) as lat:
        if lanes:
            lat.set_lanes(lanes)
        lat.set_links(links)
        lat.half_sweep(mu, parity)
        return lat.get_links()


def touched(L, site, nu, mu, parity):
    """Boolean [x3, x2, x1, x0]: sites of `parity` whose update of U_mu reads the link U_nu(site)."""
    hit = np.zeros((L[3], L[2], L[1], L[0]), dtype=bool)

    def mark(*steps):
        x = list(site)
        for d, e in steps:
            x[d] = (x[d] + e) % L[d]
        if sum(x) % 2 == parity:
            hit[x[3], x[2], x[1], x[0]] = True

    if nu == mu:
        mark()
        for d in range(4):
            if d != mu:
                mark((d, 1))
                mark((d, -1))
    else:  # U_nu at x, x + mu, x - nu, x + mu - nu
        mark()
        mark((mu, -1))
        mark((nu, 1))
        mark((nu, 1), (mu, -1))
    return hit


@pytest.mark.parametrize("kind", ["stretched", "nan", "inf", "huge", "zero"])
@pytest.mark.parametrize("lanes,decomp", [(1, None), (4, None), (0, (2, 2, 1))])
def test_one_far_link_takes_fp64_arithmetic_everywhere_else_equal(kind, lanes, decomp):
    # One link far from SU(3) sends the whole lattice through the FP64 update;
    # links that do not read it agree with the proper configuration's update,
    # links that do see it as it is.  1e-12: the bound of the parity tests.
    L = (8, 4, 6, 4)
    ref = oracle.hot_start(L, 5)
    bad = ref.copy()
    site, nu = (1, 2, 3, 0), 1
    at = (site[3], site[2], site[1], site[0], nu)
    if kind == "stretched":
        bad[at] *= 1.5
    else:
        bad[at] = {"nan": np.nan, "inf": np.inf, "huge": 1e200, "zero": 0.0}[kind]
    for mu in range(4):
        parity = (sum(site) + (mu != nu)) % 2
        a = half_sweep(L, ref, mu, parity, lanes, decomp)
        b = half_sweep(L, bad, mu, parity, lanes, decomp)
        hit = touched(L, site, nu, mu, parity)
        same = ~hit
        diff = np.abs(a[..., mu, :, :, :] - b[..., mu, :, :, :]).max(axis=(-1, -2, -3))
        assert diff[same].max() <= 1e-12
        if kind == "nan":
            # a staple that is not a number is no reason to change a link: its
            # subgroups are left, like those of a degenerate staple
            if mu == nu:
                assert np.isnan(b[at]).any()
                hit[site[3], site[2], site[1], site[0]] = False
            still = np.abs(b[..., mu, :, :, :] - ref[..., mu, :, :, :]).max(axis=(-1, -2, -3))
            assert (still[hit] <= 1e-12).all()
        elif kind == "stretched":
            assert np.isfinite(b).all()
            assert diff[hit].max() > 1e-6


def test_nan_stays_where_it_is():
    # A NaN link keeps the sweeps in FP64 arithmetic, also after the first one:
    # it stays NaN, the links that read it stay, and nothing else is lost.
    L = (8, 8, 4, 4)
    ref = oracle.hot_start(L, 5)
    bad = ref.copy()
    bad[0, 0, 0, 0, 2] = np.nan
    with su3.Lattice(L, BETA, 3, start=su3.SU3_COLD) as lat:
        lat.set_links(bad)
        lat.sweep(3)
        u = lat.get_links()
    lost = np.isnan(u).any(axis=(-1, -2, -3))
    assert lost.sum() == 1 and lost[0, 0, 0, 0, 2]
    for mu in range(4):
        frozen = touched(L, (0, 0, 0, 0), 2, mu, 0) | touched(L, (0, 0, 0, 0), 2, mu, 1)
        frozen[0, 0, 0, 0] &= mu != 2
        assert np.abs(u - ref)[..., mu, :, :, :].max(axis=(-1, -2, -3))[frozen].max() <= 1e-12


@pytest.mark.parametrize("lanes", [1, 4])
def test_links_of_fp32_accuracy_are_reunitarised(lanes):
    # Links unitary to 1e-7 only (an FP32 configuration): the update's first
    # order reunitarisation does not reach that far, its FP64 Gram-Schmidt
    # does.  Against the oracle to 1e-5 (the staples differ by the links'
    # distance from SU(3), times at most 6 |A| ~ 40 through the heatbath).
    L = (4, 6, 4, 8)
    rough = oracle.hot_start(L, 9).astype(np.float32).astype(np.float64)
    got = half_sweep(L, rough, 2, 1, lanes)
    ref = rough.copy()
    oracle.half_sweep(L, BETA, 3, 0, 2, 1, ref)
    changed = (got != rough).any(axis=(-1, -2, -3))
    assert changed.sum() == np.prod(L) // 2 and changed[..., 2].sum() == changed.sum()
    u = (got[..., 0] + 1j * got[..., 1])[changed]
    assert np.abs(u @ u.conj().transpose(0, 2, 1) - np.eye(3)).max() <= 1e-14
    assert np.abs(np.linalg.det(u) - 1).max() <= 1e-14
    off = np.abs(got - ref).max(axis=(-1, -2, -3))
    assert (off > 1e-5).sum() <= 1  # an accept decision at its threshold


def test_near_identity_and_zero_entries():
    # Exact ones and zeros (the cold start), and a configuration close to it.
    L = (4, 4, 4, 4)
    for beta in (5.7, 1e6):
        ref = oracle.cold_start(L)
        oracle.sweep(L, beta, 3, 0, 2, ref)
        with su3.Lattice(L, beta, 3, start=su3.SU3_COLD) as lat:
            lat.sweep(2)
            assert np.abs(lat.get_links() - ref).max() <= 1e-12


@pytest.mark.parametrize("L", [(2, 2, 2, 2), (4, 4, 4, 4), (6, 4, 10, 8), (8, 8, 8, 16), (10, 14, 6, 12)])
@pytest.mark.parametrize("tries", [1, 6])
def test_lanes_share_an_update_bit_for_bit(L, tries):
    # One, four and the automatic number of lanes per link (eight up to 8^4), and
    # batches (one lane, other launches): integer sums, so the same bits; the
    # same acceptance counts.
    got = []
    for lanes in (1, 4, 0):
        with su3.Lattice(L, BETA, 17, start=su3.SU3_HOT) as lat:
            lat.set_lanes(lanes)
            lat.set_heatbath(tries)
            lat.set_stats(True)
            lat.sweep(2)
            lat.half_sweep(3, 1)
            got.append((lat.get_links(), lat.stats()))
    for links, stats in got[1:]:
        assert np.array_equal(links, got[0][0])
        assert stats == got[0][1]
    with su3.Lattice(L, BETA, 17, start=su3.SU3_HOT) as lat, \
            su3.Batch([L, (4, 4, 4, 4)], [BETA, 6.0], [17, 5], start=su3.SU3_HOT, precision=su3.SU3_FP64) as bt:
        lat.set_heatbath(tries)
        bt.set_heatbath(tries)
        lat.sweep(2)
        bt.sweep(2)
        assert np.array_equal(lat.get_links(), bt.get_links(0))
        assert lat.plaquette() == bt.plaquettes()[0]


@pytest.mark.parametrize("L", [(2, 2, 2, 2), (6, 4, 10, 8), (2, 6, 2, 10), (16, 16, 16, 16)])
def test_plaquette_of_proper_and_far_configurations(L):
    # 1e-14: a sum of 6 V terms of at most 1e-15 each over 6 V (the parity tests' bound is 1e-13)
    ref = oracle.hot_start(L, 8)
    far = ref.copy()
    far[0, 0, 0, 0, 1] *= 3.0
    lost = ref.copy()
    lost[0, 0, 0, 0, 1] = np.nan
    with su3.Lattice(L, BETA, 3, start=su3.SU3_COLD) as lat:
        assert lat.plaquette() == 1.0
        lat.set_links(ref)
        assert abs(lat.plaquette() - oracle.plaquette(L, ref)) <= 1e-14
        lat.set_links(far)
        assert abs(lat.plaquette() - oracle.plaquette(L, far)) <= 1e-14
        lat.set_links(lost)
        assert np.isnan(su3.load_library().su3_plaquette(lat.handle))
        lat.set_links(ref)
        assert abs(lat.plaquette() - oracle.plaquette(L, ref)) <= 1e-14


@pytest.mark.parametrize("L", [(6, 6, 6, 4), (14, 14, 14, 8), (16, 16, 16, 16)])
@pytest.mark.parametrize("prec", [su3.SU3_FP32_MIXED, su3.SU3_FP32_EFT])
def test_fp32_one_thread_per_link_of_a_paired_store(L, prec):
    # Small site-paired lattices run one thread per link; measuring sweeps run one
    # thread per pair: the same chain, bit for bit.
    with su3.Lattice(L, BETA, 23, precision=prec) as a, su3.Lattice(L, BETA, 23, precision=prec) as b:
        a.set_lanes(1)
        b.set_lanes(1)
        a.sweep(2)
        b.sweep_measured(2)
        assert np.array_equal(a.get_links(), b.get_links())
