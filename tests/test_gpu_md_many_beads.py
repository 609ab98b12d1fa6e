"""MD of a few particles with as many beads as the launch of the pair forces takes
(65,535), with friction: the thermostat's blocks share that launch.

Reference: the MD oracle, one step.  Tolerance: springs and kicks are a few
float64 (mixed: float32) roundings of numbers no larger than the largest
velocity, 1e-12 (1e-5) of it, as in the other MD tests of one step.
"""
import numpy as np
import pytest
import torch

import oracle
from paper_2305_18025_gb300 import inputs
from paper_2305_18025_gb300.exchange import RingPolymerMD

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("P", [64321, 65535])
@pytest.mark.parametrize("prec,tol", [("fp64", 1e-12), ("mixed", 1e-5)])
def test_one_step_with_friction(P, prec, tol):
    N, beta, dt, kw = 2, 1.0, 1e-4, dict(omega0=1.0, seed=9)
    wP = inputs.omega_P(P, beta)
    rng = np.random.default_rng(P)
    pos = rng.normal(0.0, 1.0, (N, 1, 3)) + 0.003 * rng.normal(0.0, 1.0, (N, P, 3))
    vel = rng.normal(0.0, 1.0, (N, P, 3))
    ox, ov, _ = oracle.long_double.md_run(pos.copy(), vel.copy(), 1.0, wP, beta, dt, 1.0, 1, pair_type=1, pair_a=3.0,
                                          pair_b=0.5, **kw)
    md = RingPolymerMD(N, P, 1.0, wP, beta, dt=dt, gamma=1.0, gaussian=(3.0, 0.5), precision=prec, **kw)
    x, v = torch.from_numpy(pos.copy()).cuda(), torch.from_numpy(vel.copy()).cuda()
    md.step(x, v, 1)
    md.close()
    assert np.abs(x.cpu().numpy() - ox).max() <= tol * np.abs(ox).max()
    assert np.abs(v.cpu().numpy() - ov).max() <= tol * np.abs(ov).max()
