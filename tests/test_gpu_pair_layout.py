"""Stored pair factors of systems on the recursion clusters (four rows by all
sources), at every remainder of N modulo 4 and at the edges of the row tiles,
against the long-double oracle; tolerances as in test_gpu_exterior.py (FP64:
recursions within N 2^-51 in the worst case; mixed: float32 bead differences),
and for the connection probabilities those of test_gpu_recompute.py.
"""
import numpy as np
import pytest
import torch

import oracle
from paper_2305_18025_gb300 import inputs
from paper_2305_18025_gb300.exchange import ExchangeEnergy

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [129, 130, 131, 132, 159, 160, 161, 1026])
def test_stored_factors_at_every_remainder(N):
    P, beta = 3, 1.3
    wP = inputs.omega_P(P, beta)
    pos = inputs.clustered_chain_positions(N, P, seed=90 + N)
    V, F, Vf, Vb, M = oracle.long_double.fast_pimdb(pos, 1.0, wP, beta, full=True)
    for prec, tol, mtol in (("fp64", 1e-12, 1e-10), ("mixed", 1e-6, 1e-5), ("mixed32", 1e-5, 1e-5)):
        eng = ExchangeEnergy(N, P, 1.0, wP, beta, precision=prec)
        Vg, Fg = eng.forces(torch.from_numpy(pos).cuda())
        eng.sync()
        Vfg, Vbg, _ = eng.potentials()
        Mg = eng.connection_probabilities().cpu().numpy()
        eng.close()
        assert abs(float(Vg) - float(V)) <= tol * max(abs(float(V)), 1.0 / beta), prec
        assert np.linalg.norm(Fg.cpu().numpy() - np.asarray(F, np.float64)) <= tol * np.linalg.norm(F), prec
        np.testing.assert_allclose(Vfg, np.asarray(Vf, np.float64), rtol=tol, atol=tol / beta)
        np.testing.assert_allclose(Vbg, np.asarray(Vb, np.float64), rtol=tol, atol=tol / beta)
        np.testing.assert_allclose(Mg, np.asarray(M, np.float64), rtol=0, atol=mtol)
