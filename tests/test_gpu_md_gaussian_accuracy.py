"""Float64 Gaussian pair forces of the MD step, each relative to its own terms:
isolated pairs, Gaussians far wider and far narrower than the system, nearly
coincident particles, and systems that are flat along one axis.

One noiseless step of dt = 2^-60 from rest leaves the positions unchanged and
makes v = dt F without rounding; springs of frequency 1e-150 put the exchange
force at 1e-300.  The reference is the plain sum in long double.

Tolerance, in units of 2^-53 of sum |e d| per component: the exponent
a = d^2 / (2 s^2) carries at most four roundings of its own size (1/s^2, the
constant, d^2), each changing e by a; the power, the product, the conversion and
addition of eight partial sums, the force constant, 1/P and the kicks add at most
sixteen.  U-bar counts each particle's own e = 1 and subtracts it: N 2^-50 g.
"""
import numpy as np
import pytest
import torch

from paper_2305_18025_gb300.exchange import BatchedExchangeEnergy, RingPolymerMD

pytestmark = pytest.mark.gpu
LD = np.longdouble
DT = 2.0 ** -60


def reference(pos, g, s):
    """Per bead slice: forces, their error unit sum (16 + 4 a) |e d| g / s^2, U-bar."""
    N, P, _ = pos.shape
    F, unit, U = np.zeros(pos.shape, LD), np.zeros(pos.shape, LD), LD(0)
    for j in range(P):
        r = pos[:, j].astype(LD)
        d = r[:, None] - r[None]
        with np.errstate(under="ignore"):
            a = (d * d).sum(2) / (2 * LD(s)) / LD(s)
            e = np.exp(-a) * (1 - np.eye(N, dtype=LD))
            t = e[..., None] * d * (LD(g) / LD(s) / LD(s))
            F[:, j] = t.sum(1) / P
            unit[:, j] = (np.abs(t) * (16 + 4 * a)[..., None]).sum(1) / P
        U += LD(g) * e.sum() / 2 / P
    return F, unit, U


def positions(kind, N):
    rng = np.random.default_rng(11)
    if kind.startswith("pair"):  # two particles `pair<multiple of s>` apart, off the axes
        d = float(kind[4:]) * 0.5 * np.array([0.6, -0.64, 0.48])
        return np.stack([np.tile(-0.5 * d, (2, 1)), np.tile(0.5 * d, (2, 1))]) + 0.25
    pos = rng.uniform(-2.0, 2.0, (N, 2, 3))
    if kind == "flat":
        pos[..., 2] *= 1e-6
    if kind == "plane":
        pos[..., 2] = 0.0
    if kind == "sparse":
        pos *= 8.0
    if kind == "close":  # neighbours 1e-10 apart
        pos = 1.0 + rng.uniform(-1e-10, 1e-10, (N, 2, 3))
    if kind == "far":  # close pairs, far from the origin and from each other
        pos = np.repeat(rng.uniform(-60.0, 60.0, (N // 2, 2, 3)), 2, 0) + rng.uniform(-1e-5, 1e-5, (N, 2, 3))
    return pos


CASES = [("pair3", 2, 0.5), ("pair6", 2, 0.5), ("pair9", 2, 0.5), ("pair20", 2, 0.5), ("pair0", 2, 0.5), ("flat", 65, 0.5),
         ("plane", 33, 0.5), ("sparse", 40, 0.5), ("close", 33, 0.5), ("far", 34, 0.5), ("wide", 64, 0.05),
         ("wide", 64, 0.5), ("wide", 64, 50.0), ("wide", 64, 5e3), ("wide", 64, 5e5), ("wide", 64, 1e10),
         ("wide", 33, 1e160), ("many", 1027, 0.5)]


@pytest.mark.parametrize("kind,N,s", CASES)
def test_pair_forces_relative_to_their_own_size(kind, N, s):
    pos, g, P = positions(kind, N), 3.0, 2
    F, unit, U = reference(pos, g, s)
    md = RingPolymerMD(N, P, 1.0, 1e-150, 1.0, dt=DT, gamma=0.0, gaussian=(g, s))
    x, v = torch.from_numpy(pos.copy()).cuda(), torch.zeros((N, P, 3), dtype=torch.float64, device="cuda")
    en = md.step(x, v, 1).cpu().numpy()
    md.close()
    assert np.array_equal(x.cpu().numpy(), pos)
    got = v.cpu().numpy().astype(LD) / LD(DT)
    assert (np.abs(got - F) <= unit * LD(2.0) ** -53 + LD(1e-290)).all(), \
        float((np.abs(got - F) / (unit * LD(2.0) ** -53 + LD(1e-290))).max())
    assert abs(LD(en[1]) - U) <= N * 2.0 ** -50 * g + U * LD(2.0) ** -50


def test_powers_near_the_end_of_the_float64_range():
    pos, g, s = positions("pair37", 2), 1e200, 0.5  # e = 2^-987
    F, unit, _ = reference(pos, g, s)
    md = RingPolymerMD(2, 2, 1.0, 1e-150, 1.0, dt=DT, gamma=0.0, gaussian=(g, s))
    x, v = torch.from_numpy(pos.copy()).cuda(), torch.zeros((2, 2, 3), dtype=torch.float64, device="cuda")
    md.step(x, v, 1)
    md.close()
    assert (np.abs(v.cpu().numpy().astype(LD) / LD(DT) - F) <= unit * LD(2.0) ** -53).all()


def test_replicas_take_the_same_pairs():
    kinds = [("pair9", 2, 0.5), ("flat", 65, 0.5), ("close", 33, 0.5)]
    g, s = 3.0, 0.5
    ps = [positions(k, n) for k, n, _ in kinds]
    eng = BatchedExchangeEnergy([len(p) for p in ps], [2] * 3, 1.0, [1e-150] * 3, [1.0] * 3,
                                md=dict(dt=DT, gamma=0.0, gaussian=(g, s)))
    x = eng.pack([torch.from_numpy(p) for p in ps])
    v = torch.zeros_like(x)
    eng.step(x, v, 1)
    for p, w in zip(ps, eng.unpack(v)):
        F, unit, _ = reference(p, g, s)
        assert (np.abs(w.cpu().numpy().astype(LD) / LD(DT) - F) <= unit * LD(2.0) ** -53 + LD(1e-290)).all()
    eng.close()
