"""MD of systems whose recursions run in several superblocks, with the physical
force and the thermostat beside them: steps launched one by one (legacy default
stream) and replayed as a graph, against the MD oracle.  Tolerances as in
test_gpu_md.py (1e-10, mixed forms 1e-5).
"""
import functools

import numpy as np
import pytest
import torch

import oracle
from paper_2305_18025_gb300 import inputs
from paper_2305_18025_gb300.exchange import RingPolymerMD

pytestmark = pytest.mark.gpu
P, BETA, STEPS = 2, 1.0, 3


@functools.lru_cache(None)
def reference(N):
    pos = inputs.trapped_positions(N, P, N)
    vel = np.random.default_rng(N).normal(0.0, 0.5, pos.shape)
    out = oracle.float64.md_run(pos, vel, 1.0, inputs.omega_P(P, BETA), BETA, 0.01, 1.0, STEPS, omega0=1.0,
                                pair_type=1, pair_a=3.0, pair_b=0.5, seed=7)
    return pos, vel, out


@pytest.mark.parametrize("N,recompute", [(1100, True), (1800, False), (2100, True), (2800, False)])
@pytest.mark.parametrize("graph", [False, True])
@pytest.mark.parametrize("prec,tol", [("fp64", 1e-10), ("mixed", 1e-5)])
def test_trajectory(N, recompute, graph, prec, tol):
    pos, vel, (ox, ov, oe) = reference(N)
    md = RingPolymerMD(N, P, 1.0, inputs.omega_P(P, BETA), BETA, dt=0.01, gamma=1.0, omega0=1.0, gaussian=(3.0, 0.5),
                       seed=7, precision=prec, recompute=recompute, stream=torch.cuda.Stream() if graph else None)
    x, v = torch.from_numpy(pos.copy()).cuda(), torch.from_numpy(vel.copy()).cuda()
    torch.cuda.synchronize()
    en = md.step(x, v, STEPS).cpu().numpy()
    md.close()
    assert np.abs(x.cpu().numpy() - ox).max() <= tol * np.abs(ox).max()
    assert np.abs(v.cpu().numpy() - ov).max() <= tol * np.abs(ov).max()
    np.testing.assert_allclose(en, oe, rtol=0, atol=tol * np.abs(oe).max())
