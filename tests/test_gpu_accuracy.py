"""How exact the FP64 link update is: half-sweeps on the GPU against the same update in numpy's long double (113 bits
on AArch64, 64 on x86), in units of 2^-53, next to the FP64 oracle on the same links.

The link-by-link parity tests stop at 1e-12, thousands of such units; here an FP32 remainder or a series
coefficient that is slightly off would show.
"""
import numpy as np
import pytest

import oracle
import paper_0904_1179_gb300 as su3

pytestmark = pytest.mark.gpu

LD = np.longdouble
U53 = 2.0 ** -53


def philox(site, w1, w2, w3, seed):
    m32 = np.uint64(0xFFFFFFFF)
    c = [site.astype(np.uint64)] + [np.full(site.shape, w, np.uint64) for w in (w1, w2, w3)]
    k0, k1 = seed & 0xFFFFFFFF, seed >> 32
    for _ in range(10):
        a, b = c[0] * np.uint64(0xD2511F53), c[2] * np.uint64(0xCD9E8D57)
        c = [(b >> np.uint64(32)) ^ c[1] ^ np.uint64(k0), b & m32, (a >> np.uint64(32)) ^ c[3] ^ np.uint64(k1), a & m32]
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    return c


def uniforms(site, mu, sub, seed):
    out = []
    for call in range(3):
        w = philox(site, mu | sub << 2 | call << 4, 0, 0, seed)
        for q in (0, 2):
            m = (w[q] << np.uint64(21)) | ((w[q + 1] >> np.uint64(12)) << np.uint64(1)) | np.uint64(1)
            out.append(m.astype(LD) * LD(2.0) ** -53)
    return out


def dagger(a):
    return a.conj().swapaxes(-1, -2)


def reference_half_sweep(L, beta, seed, mu, parity, links):
    """The links U_mu(x) of parity `parity` after their update at sweep 0 (sites in storage order), the sites' mask,
    and which of them count: every projection at least a third of its largest value 12, no accept decision
    within 1e-12 of its threshold."""
    U = links[..., 0].astype(LD) + LD(1) * 1j * links[..., 1].astype(LD)

    def link(nu, *steps):
        a = U[..., nu, :, :]
        for d, e in steps:
            a = np.roll(a, -e, axis=3 - d)
        return a

    A = 0
    for nu in range(4):
        if nu != mu:
            A = A + link(nu, (mu, 1)) @ dagger(link(mu, (nu, 1))) @ dagger(link(nu))
            A = A + dagger(link(nu, (mu, 1), (nu, -1))) @ dagger(link(mu, (nu, -1))) @ link(nu, (nu, -1))
    site = np.arange(np.prod(L)).reshape(L[3], L[2], L[1], L[0])
    x3, x2, x1, x0 = np.indices(site.shape)
    here = (x0 + x1 + x2 + x3) % 2 == parity
    A, u, s = A[here], link(mu)[here].copy(), site[here]
    counts = np.ones(len(s), bool)
    two_pi = 2 * np.arccos(LD(-1))
    for sub, (i, j) in enumerate(((0, 1), (0, 2), (1, 2))):
        W = u @ A
        r = np.stack([(W[:, i, i] + W[:, j, j]).real, (W[:, i, j] + W[:, j, i]).imag,
                      (W[:, i, j] - W[:, j, i]).real, (W[:, i, i] - W[:, j, j]).imag], -1)
        k2 = np.sqrt((r * r).sum(-1))
        v = r / k2[:, None]
        u0, u1, u2, u3, u4, u5 = uniforms(s, mu, sub, seed)
        delta = -(np.log(u0) + np.cos(two_pi * u1) ** 2 * np.log(u2)) * 3 / (LD(beta) * k2)
        margin = 1 - delta / 2 - u3 * u3
        counts &= (k2 >= 4) & (np.abs(margin) > 1e-12)
        ok = margin >= 0
        rho = np.sqrt(np.maximum(delta * (2 - delta), 0))
        ct, sn = 1 - 2 * u4, 2 * np.sqrt(u4 * (1 - u4))
        a = np.stack([1 - delta, rho * sn * np.cos(two_pi * u5), rho * sn * np.sin(two_pi * u5), rho * ct], -1)

        def matrix(q):
            return np.stack([q[:, 0] + 1j * q[:, 3], q[:, 2] + 1j * q[:, 1],
                             -q[:, 2] + 1j * q[:, 1], q[:, 0] - 1j * q[:, 3]], -1).reshape(-1, 2, 2)

        rows = (matrix(a) @ dagger(matrix(v))) @ u[:, [i, j], :]
        u[:, [i, j], :] = np.where(ok[:, None, None], rows, u[:, [i, j], :])
    a, b = u[:, 0], u[:, 1]
    a = a / np.sqrt((np.abs(a) ** 2).sum(-1, keepdims=True))
    b = b - (a.conj() * b).sum(-1, keepdims=True) * a
    b = b / np.sqrt((np.abs(b) ** 2).sum(-1, keepdims=True))
    c = np.stack([a[:, (k + 1) % 3] * b[:, (k + 2) % 3] - a[:, (k + 2) % 3] * b[:, (k + 1) % 3] for k in range(3)], -1)
    u = np.stack([a, b, c.conj()], -2)
    return np.stack([u.real, u.imag], -1), here, counts


def configuration(L, kind):
    if kind == "cold":
        return oracle.cold_start(L), 5.7
    if kind == "hot":
        return oracle.hot_start(L, 4), 5.7
    beta = float(kind)
    with su3.Lattice(L, beta, 9, start=su3.SU3_COLD) as lat:
        lat.sweep(12)
        return lat.get_links(), beta


@pytest.mark.parametrize("kind", ["cold", "hot", "5.7", "50", "1000"])
@pytest.mark.parametrize("mu,parity", [(0, 0), (2, 1)])
def test_half_sweep_errors(kind, mu, parity):
    L, seed = (8, 4, 4, 6), (7 << 32) + 3
    links, beta = configuration(L, kind)
    want, here, counts = reference_half_sweep(L, beta, seed, mu, parity, links)
    assert kind == "hot" or counts.mean() > 0.9
    plain = links.copy()
    oracle.half_sweep(L, beta, seed, 0, mu, parity, plain)

    def errors(got):
        return ((got[..., mu, :, :, :][here] - want)[counts] / U53).astype(float)

    fp64 = np.sqrt((errors(plain) ** 2).mean())
    for lanes, decomp in ((1, None), (4, None), (0, None), (0, (2, 2, 1))):
        with su3.Lattice(L, beta, seed, start=su3.SU3_COLD, decomp=decomp) as lat:
            if lanes:
                lat.set_lanes(lanes)
            lat.set_links(links)
            lat.half_sweep(mu, parity)
            e = errors(lat.get_links())
        # A staple entry is good to 4 units, so a projection (rows of norm 1, three columns, two rows) to 4 * 2 sqrt(3),
        # its direction at |2r| >= 4 to 3.5; the proposal and the rotation add up to 4 more; three subgroups, and 4
        # for the reunitarisation: 27 at most.  On average no more than in FP64 arithmetic.
        assert np.abs(e).max() <= 27.0, (lanes, decomp)
        assert np.sqrt((e ** 2).mean()) <= fp64, (lanes, decomp)
