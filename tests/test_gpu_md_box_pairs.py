"""All-pairs forces of the MD step in a periodic box (boxes of fewer than three
cutoffs a side take no cell lists), at the edges of the blocks of particles.

One noiseless step of dt = 2^-60 from rest makes v = dt F without rounding;
springs of frequency 1e-150 put the exchange force at 1e-300.  The reference is
the plain minimum-image sum in long double.

Tolerance, float64: a difference is rounded twice at the size of the box, so to
2^-52 L, and a pair's force changes by at most 14 (Lennard-Jones, whose terms go as
r^-14) or 1 + 2a (Gaussian, a = d^2 / 2 s^2) times that over r; beside it at most 64
roundings of a term (powers of a quotient, sums, constants): 2^-53 (64 + 28 L / r)
and 2^-53 (64 + 4 a + 2 (1 + 2 a) L / |d|) of each term.  Mixed: the same count
of float32 roundings.
"""
import numpy as np
import pytest
import torch

from paper_2305_18025_gb300.exchange import RingPolymerMD

pytestmark = pytest.mark.gpu
LD = np.longdouble
DT = 2.0 ** -60
L, SIG, RC, EPS = 6.0, 0.8, 2.9, 1.0
G, S = 3.0, 0.5


def lattice(N, P):
    """Particles apart from one another, scattered over several images of the box."""
    rng = np.random.default_rng(N)
    k = int(np.ceil(N ** (1.0 / 3.0)))
    cells = np.array([(i, j, m) for i in range(k) for j in range(k) for m in range(k)], float)[:N]
    pos = (cells[:, None] + 0.5 + rng.uniform(-0.15, 0.15, (N, P, 3))) * (L / k)
    return pos + L * rng.integers(-2, 3, (N, 1, 3))


def reference(pos, lj):
    N, P, _ = pos.shape
    F, unit, U = np.zeros(pos.shape, LD), np.zeros(pos.shape, LD), LD(0)
    off = ~np.eye(N, dtype=bool)
    for j in range(P):
        r = pos[:, j].astype(LD)
        d = r[:, None] - r[None]
        d -= LD(L) * np.rint(d / LD(L))
        r2 = np.where(off, (d * d).sum(2), LD(1))
        ratio = LD(L) / np.sqrt(r2)
        if lj:
            on = off & (r2 < LD(RC) * LD(RC))
            s6 = np.where(on, (LD(SIG) * LD(SIG) / r2) ** 3, LD(0))
            c6 = (LD(SIG) / LD(RC)) ** 6
            f = 24 * LD(EPS) * (2 * s6 * s6 - s6) / r2
            mag = 24 * LD(EPS) * (2 * s6 * s6 + s6) / r2 * (64 + 28 * ratio)
            U += (4 * LD(EPS) * ((s6 * s6 - s6) - on * (c6 * c6 - c6))).sum() / 2 / P
        else:
            a = r2 / (2 * LD(S) * LD(S))
            f = np.where(off, np.exp(-a), LD(0)) * LD(G) / LD(S) / LD(S)
            mag = f * (64 + 4 * a)
            U += f.sum() * LD(S) * LD(S) / 2 / P
        F[:, j] = (f[..., None] * d).sum(1) / P
        unit[:, j] = (mag[..., None] * np.abs(d)).sum(1) / P
        if not lj:
            unit[:, j] += (f * 2 * (1 + 2 * a) * LD(L))[..., None].repeat(3, 2).sum(1) / P
        else:
            unit[:, j] += (np.abs(f) * 28 * LD(L))[..., None].repeat(3, 2).sum(1) / P
    return F, unit, U


@pytest.mark.parametrize("N", [2, 15, 16, 17, 33, 65])
@pytest.mark.parametrize("lj", [False, True])
@pytest.mark.parametrize("prec,u", [("fp64", -53), ("mixed", -24)])
def test_all_pairs_in_a_box(N, lj, prec, u):
    pos = lattice(N, 2)
    F, unit, U = reference(pos, lj)
    kw = dict(lennard_jones=(EPS, SIG, RC)) if lj else dict(gaussian=(G, S))
    md = RingPolymerMD(N, 2, 1.0, 1e-150, 1.0, dt=DT, gamma=0.0, precision=prec, box=L, **kw)
    x, v = torch.from_numpy(pos.copy()).cuda(), torch.zeros((N, 2, 3), dtype=torch.float64, device="cuda")
    en = md.step(x, v, 1).cpu().numpy()
    md.close()
    got = v.cpu().numpy().astype(LD) / LD(DT)
    # mixed: a float32 coordinate of up to three boxes is rounded at 2^-24 of itself
    worst = (np.abs(got - F) / (unit * (1 if prec == "fp64" else 3) * LD(2.0) ** u + LD(1e-290))).max()
    assert worst <= 1, float(worst)
    assert abs(LD(en[1]) - U) <= LD(2.0) ** u * (unit.sum() * L + N)
