"""Lennard-Jones forces by cell lists where every particle has ~90 partners inside
the cutoff, so that the float64 kernel's list of 32 near candidates is worked off
inside the loop, several times, before the rest at its end.

One noiseless step of dt = 2^-60 from rest makes v = dt F without rounding; springs
of frequency 1e-150 put the exchange force at 1e-300.  Reference and tolerance as in
test_gpu_md_box_pairs.py: 2^-53 (2^-24 mixed) times 64 + 28 L / r of each term.
"""
import numpy as np
import pytest
import torch

from paper_2305_18025_gb300.exchange import RingPolymerMD

pytestmark = pytest.mark.gpu
LD = np.longdouble
DT = 2.0 ** -60
L, SIG, RC, EPS, K = 9.0, 0.6, 2.95, 1.0, 9  # a jittered lattice of K^3 sites, 3 cells a side


@pytest.mark.parametrize("prec,u", [("fp64", -53), ("mixed", -24)])
def test_lists_are_worked_off_as_they_fill(prec, u):
    N, P = K ** 3, 2
    rng = np.random.default_rng(2)
    cells = np.stack(np.meshgrid(*3 * [np.arange(K)], indexing="ij"), -1).reshape(-1, 1, 3)
    pos = (cells + 0.5 + rng.uniform(-0.2, 0.2, (N, P, 3))) * (L / K) + L * rng.integers(-1, 2, (N, 1, 3))
    F, unit, U = np.zeros(pos.shape, LD), np.zeros(pos.shape, LD), LD(0)
    off = ~np.eye(N, dtype=bool)
    for j in range(P):
        r = pos[:, j].astype(LD)
        d = r[:, None] - r[None]
        d -= LD(L) * np.rint(d / LD(L))
        r2 = np.where(off, (d * d).sum(2), LD(1))
        on = off & (r2 < LD(RC) * LD(RC))
        assert on.sum(1).min() > 64
        s6 = np.where(on, (LD(SIG) * LD(SIG) / r2) ** 3, LD(0))
        c6 = (LD(SIG) / LD(RC)) ** 6
        U += (4 * LD(EPS) * ((s6 * s6 - s6) - on * (c6 * c6 - c6))).sum() / 2 / P
        f, mag = 24 * (2 * s6 * s6 - s6) / r2, 24 * (2 * s6 * s6 + s6) / r2
        F[:, j] = (f[..., None] * d).sum(1) / P
        unit[:, j] = (mag[..., None] * ((64 + 28 * LD(L) / np.sqrt(r2))[..., None] * np.abs(d) + 28 * LD(L))).sum(1) / P
    md = RingPolymerMD(N, P, 1.0, 1e-150, 1.0, dt=DT, gamma=0.0, precision=prec, box=L, lennard_jones=(EPS, SIG, RC))
    x, v = torch.from_numpy(pos.copy()).cuda(), torch.zeros((N, P, 3), dtype=torch.float64, device="cuda")
    en = md.step(x, v, 1).cpu().numpy()
    md.close()
    got = v.cpu().numpy().astype(LD) / LD(DT)
    worst = (np.abs(got - F) / (unit * LD(2.0) ** u)).max()
    assert worst <= 1, float(worst)
    assert abs(LD(en[1]) - U) <= LD(2.0) ** u * (unit.sum() * L + N)
