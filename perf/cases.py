"""What a user of this library has it do, as cases that can be timed and checked.

A case is one pass through the public entry points: heatbath sweeps of a
lattice (or of a batch of replicas) followed by what a simulation program does
with the result -- the configuration fetched into its own page-locked buffer,
with the plaquettes it measured.  `listed()` are the sizes of the package's
workloads (the columns of Table 1 of Berg & Wu, arXiv:0904.1179, the 48^4
precision study, the 96-replica batch) and a few of ragged extents; `draw()`
gives others of the same ranges.  `exact()` is the same pass in plain torch,
64 bits.

A chain is chaotic: two that differ by rounding separate by about a factor of
two per sweep, and an accept decision that flips changes a whole link.  FP64
cases therefore run few sweeps per pass, and `exact()` has a value for FP32
chains of one or two sweeps only.
"""
import math

import numpy as np
import torch

import paper_0904_1179_gb300 as su3
from paper_0904_1179_gb300 import workloads

PRECISION = {"fp64": su3.SU3_FP64, "fp32_mixed": su3.SU3_FP32_MIXED, "fp32_eft": su3.SU3_FP32_EFT}


def _lattice(name, dims, precision, sweeps, beta=workloads.BETA, start="hot", measured=False, plaquette=False, tries=1,
             ndmpi=0, mpifactor=1, resume=False):
    return {"name": name, "kind": "lattice", "L0": dims[0], "L1": dims[1], "L2": dims[2], "L3": dims[3],
            "precision": precision, "beta": beta, "start": start, "sweeps": sweeps, "measured": measured,
            "plaquette": plaquette, "tries": tries, "ndmpi": ndmpi, "mpifactor": mpifactor, "resume": resume}


def listed():
    return [
        # the smallest call: one sweep of the 4^4 cold-start chain and its plaquette
        _lattice("4x4_fp64", (4, 4, 4, 4), "fp64", 1, start="cold", plaquette=True),
        # Table 1's columns in the plain FP64 form, a few sweeps between two configurations kept
        _lattice("8x4_fp64", (8, 8, 8, 8), "fp64", 3),
        _lattice("16x4_fp64", (16, 16, 16, 16), "fp64", 3),
        _lattice("32x4_fp64", (32, 32, 32, 32), "fp64", 2),
        # a checkpoint of the 32^4 lattice read back, two measured sweeps, the checkpoint written again
        _lattice("32x4_fp64_resume", (32, 32, 32, 32), "fp64", 2, measured=True, resume=True),
        # uneven extents with the repeat-until-accepted heatbath of the paper's non-MPI program
        _lattice("10x14x6x12_fp64_repeat", (10, 14, 6, 12), "fp64", 2, beta=6.0, tries=8),
        # the paper's domain decomposition, sixteen sublattices with the boundary exchange
        _lattice("16x4_fp64_decomposed", (16, 16, 16, 16), "fp64", 2, ndmpi=4, mpifactor=2),
        # the FP32 form where one update's latency counts, and on the headline lattice
        _lattice("8x4_fp32", (8, 8, 8, 8), "fp32_mixed", 2),
        _lattice("32x4_fp32", (32, 32, 32, 32), "fp32_mixed", 20),
        # ragged extents (the single-site FP32 layout: L3 no multiple of 4)
        _lattice("18x10x14x22_fp32", (18, 10, 14, 22), "fp32_mixed", 20),
        # the large lattice of the precision study, plaquette after every sweep
        _lattice("48x4_fp32_eft", (48, 48, 48, 48), "fp32_eft", 10, beta=6.0, measured=True),
        # 96 replicas of uneven sizes and couplings, ten sweeps between measurements
        {"name": "batch_96_fp32", "kind": "batch", "replicas": 96, "scale": 0, "precision": "fp32_mixed", "sweeps": 10},
    ]


def draw(rng):
    if rng.random() < 0.12:
        return {"kind": "batch", "replicas": rng.randint(5, 96), "scale": rng.randint(1, 1 << 20),
                "precision": rng.choice(["fp32_mixed", "fp32_eft", "fp64"]), "sweeps": rng.randint(1, 3)}
    precision = rng.choice(["fp64", "fp64", "fp32_mixed", "fp32_eft"])
    largest = 32 ** 4 if precision == "fp64" else 40 ** 4
    volume = math.exp(rng.uniform(math.log(4 ** 4), math.log(largest)))
    side = volume ** 0.25
    dims = [max(2, 2 * round(side * math.exp(rng.uniform(-0.35, 0.35)) / 2)) for _ in range(3)]
    dims.append(max(2, 2 * int(volume / (2 * dims[0] * dims[1] * dims[2]))))
    c = _lattice("", dims, precision, rng.randint(1, 2) if precision == "fp64" else rng.choice([1, 2, 8, 20]),
                 beta=round(rng.uniform(5.5, 6.2), 3))
    del c["name"]
    option = rng.randrange(6)
    if option == 0:
        c["measured"] = True
    elif option == 1:
        c["tries"] = rng.randint(2, 12)
    elif option == 2:
        # cut the directions whose extents split into even parts
        nd = 0
        while nd < 4 and dims[nd] % 4 == 0:
            nd += 1
        c["ndmpi"], c["mpifactor"] = (nd, 2) if nd else (1, 1)
    elif option == 3:
        c["resume"] = True
    elif option == 4:
        c["plaquette"] = True
    return c


def _dims(case):
    return case["L0"], case["L1"], case["L2"], case["L3"]


def _replicas(case):
    """Extents, couplings and seeds of a batch: the 96 replicas of the package's workload (as many as asked), or as
    many of uneven sizes."""
    dims, betas, seeds = workloads.batch_96()
    if case["scale"]:
        r = np.random.RandomState(case["scale"])
        dims = [tuple(int(x) for x in 2 * r.randint(2, 8, 4)) for _ in dims]
    n = case["replicas"]
    return dims[:n], betas[:n], seeds[:n]


def _pinned(n):
    """A page-locked host buffer of n doubles, as a program keeps one for its configurations."""
    return torch.zeros(n, dtype=torch.float64, pin_memory=torch.cuda.is_available()).numpy()


def prepare(case, seed):
    p = PRECISION[case["precision"]]
    if case["kind"] == "batch":
        dims, betas, seeds = _replicas(case)
        b = su3.Batch(dims, betas, [(1000003 * seed + s) & 0xFFFFFFFF for s in seeds], su3.SU3_HOT, p)
        sizes = [int(np.prod(su3.links_shape(L))) for L in dims]
        flat = _pinned(sum(sizes))
        parts, at = [], 0
        for L, n in zip(dims, sizes):
            parts.append(flat[at:at + n].reshape(su3.links_shape(L)))
            at += n
        return {"case": case, "batch": b, "links": flat, "parts": parts}
    L = _dims(case)
    decomp = (case["ndmpi"], case["mpifactor"], 1) if case["ndmpi"] else None
    lat = su3.Lattice(L, case["beta"], seed, su3.SU3_COLD if case["start"] == "cold" or case["resume"] else su3.SU3_HOT, p,
                      decomp=decomp)
    if case["tries"] > 1:
        lat.set_heatbath(case["tries"])
    state = {"case": case, "lattice": lat, "links": _pinned(int(np.prod(su3.links_shape(L)))).reshape(su3.links_shape(L))}
    if case["resume"]:
        state["saved"] = _pinned(state["links"].size).reshape(su3.links_shape(L))
        torch.from_numpy(state["saved"]).copy_(_canonical(_random_links(L, seed)))
    return state


def run(state):
    case = state["case"]
    if case["kind"] == "batch":
        b = state["batch"]
        b.sweep(case["sweeps"])
        plaquettes = b.plaquettes()
        for r, part in enumerate(state["parts"]):
            b.get_links(r, part)
        return {"plaquettes": np.array(plaquettes), "links": state["links"]}
    lat = state["lattice"]
    out = {}
    if case["resume"]:
        lat.set_links(state["saved"])
    if case["measured"]:
        out["plaquettes"] = lat.sweep_measured(case["sweeps"])
    else:
        lat.sweep(case["sweeps"])
    if case["plaquette"]:
        out["plaquette"] = lat.plaquette()
    out["links"] = lat.get_links(state["links"])
    return out


def work(case):
    """Every sweep reads and writes each link once (18 or 12 reals); the configuration comes out, and for a resumed
    chain goes in, as 18 doubles a link.  2916 operations an update, as counted on the staple of six three-link paths,
    three SU(2) steps and the reunitarisation (no transcendentals)."""
    volume = sum(int(np.prod(L)) for L in (_replicas(case)[0] if case["kind"] == "batch" else [_dims(case)]))
    links = 4 * volume
    reals = 18 * 8 if case["precision"] == "fp64" else 12 * 4
    host = 144 * links * (2 if case.get("resume") else 1)
    return {"bytes": 2 * reals * links * case["sweeps"] + host, "flops": 2916 * links * case["sweeps"]}


# ---------------------------------------------------------------------------
# The same pass in plain torch, complex numbers of 64-bit parts.  Links are
# U[mu][x3, x2, x1, x0, 3, 3].
# ---------------------------------------------------------------------------
def _device():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _unitary(rows):
    """SU(3) matrices from their rows 0 and 1 (Gram-Schmidt, row 2 = conj(row 0 x row 1))."""
    a, b = rows[..., 0, :], rows[..., 1, :]
    a = a / a.abs().square().sum(-1, keepdim=True).sqrt()
    b = b - (a.conj() * b).sum(-1, keepdim=True) * a
    b = b / b.abs().square().sum(-1, keepdim=True).sqrt()
    return torch.stack([a, b, torch.linalg.cross(a, b).conj()], -2)


def _random_links(L, seed):
    """Haar-random links from a seed."""
    g = torch.Generator(device=_device()).manual_seed(seed)
    z = torch.randn((4, L[3], L[2], L[1], L[0], 2, 3, 2), generator=g, dtype=torch.float64, device=_device())
    return _unitary(torch.view_as_complex(z))


def _canonical(U):
    """U[L3, L2, L1, L0, mu, row, column, re/im], the library's host layout."""
    return torch.view_as_real(torch.movedim(U, 0, 4).resolve_conj().contiguous())


def _mulhilo(a, m):
    """(high, low) 32-bit words of a times the constant m, in 64-bit integers (whose products have 63 bits)."""
    low = a * (m & 0xFFFF)
    high = a * (m >> 16) + (low >> 16)
    return (high >> 16) & 0xFFFFFFFF, ((high & 0xFFFF) << 16) | (low & 0xFFFF)


def _philox(site, w1, w2, w3, seed):
    """Philox4x32-10 of the counters (site, w1, w2, w3)."""
    c = [site, torch.full_like(site, w1), torch.full_like(site, w2), torch.full_like(site, w3)]
    k0, k1 = seed & 0xFFFFFFFF, (seed >> 32) & 0xFFFFFFFF
    for _ in range(10):
        h0, l0 = _mulhilo(c[0], 0xD2511F53)
        h1, l1 = _mulhilo(c[2], 0xCD9E8D57)
        c = [h1 ^ c[1] ^ k0, l1, h0 ^ c[3] ^ k1, l0]
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    return c


def _u52(a, b):
    return (((a << 20) | (b >> 12)).double() + 0.5) * 2.0 ** -52


def _u23(a):
    return ((a >> 9).double() + 0.5) * 2.0 ** -23


def _sites(L):
    shape = (L[3], L[2], L[1], L[0])
    s = torch.arange(L[0] * L[1] * L[2] * L[3], device=_device()).reshape(shape)
    x = [s % L[0], s // L[0] % L[1], s // (L[0] * L[1]) % L[2], s // (L[0] * L[1] * L[2])]
    return s, (x[0] + x[1] + x[2] + x[3]) & 1


def _round32(U):
    """Links as FP32 stores hold them: rows 0 and 1 rounded, row 2 from them."""
    a, b = U[..., 0, :].to(torch.complex64).to(torch.complex128), U[..., 1, :].to(torch.complex64).to(torch.complex128)
    return torch.stack([a, b, torch.linalg.cross(a, b).conj()], -2)


def _hot(L, seed, f32):
    site, _ = _sites(L)
    U = []
    for mu in range(4):
        z = []
        for call in range(6):
            w = _philox(site, mu | call << 4, 0, 1, seed)
            rad, ang = torch.sqrt(-2.0 * torch.log(_u52(w[0], w[1]))), 2.0 * math.pi * _u52(w[2], w[3])
            z.append(torch.complex(rad * torch.cos(ang), rad * torch.sin(ang)))
        U.append(_unitary(torch.stack(z, -1).reshape(*site.shape, 2, 3)))
    U = torch.stack(U)
    return _round32(U) if f32 else U


def _cold(L):
    eye = torch.eye(3, dtype=torch.complex128, device=_device())
    return eye.expand(4, L[3], L[2], L[1], L[0], 3, 3).clone()


def _shift(A, mu, d):
    """A(x + d mu-hat) at x."""
    return torch.roll(A, -d, dims=3 - mu)


def _half_sweep(U, mu, parity, t, beta, seed, tries, f32, site, par):
    A = 0
    for nu in range(4):
        if nu == mu:
            continue
        up, side = _shift(U[nu], mu, 1), _shift(U[mu], nu, 1)
        A = A + up @ side.mH @ U[nu].mH
        A = A + _shift(up.mH @ U[mu].mH @ U[nu], nu, -1)
    here = par == parity
    A, u, s = A[here], U[mu][here], site[here]
    for sub, (i, j) in enumerate(((0, 1), (0, 2), (1, 2))):
        W = u @ A
        r = torch.stack([(W[:, i, i] + W[:, j, j]).real, (W[:, i, j] + W[:, j, i]).imag,
                         (W[:, i, j] - W[:, j, i]).real, (W[:, i, i] - W[:, j, j]).imag], -1)  # 2r
        k2 = r.square().sum(-1).sqrt()  # 2k
        todo = k2 > 0
        a = torch.zeros_like(r)
        got = torch.zeros_like(todo)
        for n in range(tries):
            left = torch.nonzero(todo & ~got)[:, 0]
            if not len(left):
                break
            w1 = mu | sub << 2 | n << 6
            w = [_philox(s[left], w1 | call << 4, t & 0xFFFFFFFF, t >> 32 << 4, seed) for call in range(2 if f32 else 3)]
            if f32:
                u0, u1, u2, u3, u4, u5 = (_u23(x) for x in (*w[0], w[1][0], w[1][1]))
            else:
                u0, u1, u2, u3, u4, u5 = (_u52(x[q], x[q + 1]) for x in w for q in (0, 2))
            delta = -(torch.log(u0) + torch.cos(2 * math.pi * u1).square() * torch.log(u2)) * 3.0 / (beta * k2[left])
            ok = u3.square() <= 1.0 - 0.5 * delta
            a0 = 1.0 - delta
            rho = (1.0 - a0 * a0).clamp(min=0).sqrt()
            ct = 1.0 - 2.0 * u4
            sn = (1.0 - ct * ct).clamp(min=0).sqrt()
            q = torch.stack([a0, rho * sn * torch.cos(2 * math.pi * u5), rho * sn * torch.sin(2 * math.pi * u5), rho * ct], -1)
            a[left[ok]] = q[ok]
            got[left[ok]] = True
        v = r / k2.clamp(min=1e-300)[:, None]

        def m2(q):
            return torch.stack([torch.complex(q[:, 0], q[:, 3]), torch.complex(q[:, 2], q[:, 1]),
                                torch.complex(-q[:, 2], q[:, 1]), torch.complex(q[:, 0], -q[:, 3])], -1).reshape(-1, 2, 2)

        new = (m2(a) @ m2(v).mH) @ u[:, [i, j], :]
        u = u.clone()
        u[:, [i, j], :] = torch.where(got[:, None, None], new, u[:, [i, j], :])
    u = _unitary(u[:, :2, :])
    U[mu][here] = _round32(u) if f32 else u


def _plaquette(U):
    total = 0.0
    for mu in range(4):
        for nu in range(mu):
            X, Y = U[mu] @ _shift(U[nu], mu, 1), U[nu] @ _shift(U[mu], nu, 1)
            total += float((X.real * Y.real + X.imag * Y.imag).sum())
    return total / (18.0 * U[0].numel() / 9)


def exact(case, seed):
    f32 = case["precision"] != "fp64"
    if case["kind"] == "batch" or (f32 and case["sweeps"] > 2):
        return None
    L = _dims(case)
    if case["resume"]:
        U = _random_links(L, seed)
        U = _round32(U) if f32 else U
    else:
        U = _cold(L) if case["start"] == "cold" else _hot(L, seed, f32)
    site, par = _sites(L)
    plaquettes = []
    for t in range(case["sweeps"]):
        for mu in range(4):
            for parity in range(2):
                _half_sweep(U, mu, parity, t, case["beta"], seed, case["tries"], f32, site, par)
        if case["measured"]:
            plaquettes.append(_plaquette(U))
    out = {"links": _canonical(U).cpu().numpy()}
    if case["measured"]:
        out["plaquettes"] = np.array(plaquettes)
    if case["plaquette"]:
        out["plaquette"] = _plaquette(U)
    return out
