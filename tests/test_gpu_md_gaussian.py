"""Gaussian pair forces of the MD step at the edges of their blocks, chunks and
number formats, against the MD oracle (one noiseless step; from N = 128 its
long-double build, as for every parity test of that size: with centres over
+-60 the float64 build's shifted log-sum-exp is 1.3e-11 off in a velocity).

Float64 pairs run in 64-bit fixed point while |r| sqrt(log2(e) / (2 s^2)) stays
below 64, past that (scale 60 below) in float64; with a wider spread the
fixed-point unit grows.  Tolerances.  Float64: a pair's force is within 2^-54
(fixed point) or a few 2^-53 (float64) of its value, N of them add to at most
N 2^-53, i.e. 2^-43 at N = 1025, against sums of order one: 1e-12 of the largest
element.  Mixed: float32 pairs (2^-24 each, N of them) enter with dt: 1e-5.
"""
import numpy as np
import pytest
import torch

import oracle
from paper_2305_18025_gb300 import inputs
from paper_2305_18025_gb300.exchange import RingPolymerMD

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [1, 2, 31, 33, 65, 1025])
@pytest.mark.parametrize("scale", [0.3, 3.0, 12.0, 60.0])
def test_one_step_matches_the_oracle(N, scale):
    P, beta, dt, g, s = 2, 1.0, 0.01, 3.0, 0.5
    wP = inputs.omega_P(P, beta)
    rng = np.random.default_rng(N)
    pos = rng.uniform(-scale, scale, (N, 1, 3)) + rng.normal(0.0, 0.1, (N, P, 3))
    vel = rng.normal(0.0, 1.0, (N, P, 3))
    ref = oracle.long_double if N >= 128 else oracle.float64
    ox, ov, oe = ref.md_run(pos.copy(), vel.copy(), 1.0, wP, beta, dt, 0.0, 1, omega0=1.0, pair_type=1, pair_a=g,
                            pair_b=s)
    for prec, tol in (("fp64", 1e-12), ("mixed", 1e-5)):
        md = RingPolymerMD(N, P, 1.0, wP, beta, dt=dt, gamma=0.0, omega0=1.0, gaussian=(g, s), precision=prec)
        x, v = torch.from_numpy(pos.copy()).cuda(), torch.from_numpy(vel.copy()).cuda()
        en = md.step(x, v, 1).cpu().numpy()
        md.close()
        assert np.abs(x.cpu().numpy() - ox).max() <= tol * np.abs(ox).max(), prec
        # a velocity holds dt F/m, and F the exchange force k d with k = P/beta^2
        assert np.abs(v.cpu().numpy() - ov).max() <= tol * max(np.abs(ov).max(), 1.0), prec
        assert abs(en[1] - oe[1]) <= tol * max(abs(oe[1]), 1.0), prec


def test_a_non_finite_position_is_reported_and_reaches_the_velocities():
    N, P = 40, 2
    pos = np.random.default_rng(3).normal(0.0, 1.0, (N, P, 3))
    pos[7, 1, 2] = np.inf
    md = RingPolymerMD(N, P, 1.0, inputs.omega_P(P, 1.0), 1.0, dt=0.01, gamma=0.0, gaussian=(3.0, 0.5))
    x, v = torch.from_numpy(pos).cuda(), torch.zeros((N, P, 3), dtype=torch.float64, device="cuda")
    with pytest.raises(Exception):
        md.step(x, v, 1)
    assert not torch.isfinite(v[:, 1, 2]).all()
    md.close()
