"""Recomputed pair factors in a periodic box on the recursion clusters, against the
long-double oracle: one panel row past the one-CTA form (129), several panels (300),
two superblocks (1100) and three, whose later rows are added beside the recursions
(2100).  Tolerances as in test_gpu_recompute.py.
"""
import numpy as np
import pytest
import torch

import oracle
from paper_2305_18025_gb300 import inputs
from paper_2305_18025_gb300.exchange import ExchangeEnergy

pytestmark = pytest.mark.gpu
P, BETA = 4, 1.0
TOL = {"fp64": (1e-12, 1e-10), "mixed": (1e-6, 1e-5), "mixed32": (1e-6, 1e-5)}


@pytest.mark.parametrize("N", [129, 300, 1100, 2100])
def test_against_the_oracle(N):
    rng = np.random.default_rng(N)
    L = (N / 0.8) ** (1.0 / 3.0)
    # a walk through the box: neighbours overlap and cross its faces
    pos = np.mod(np.cumsum(rng.normal(0, 0.25, (N, 1, 3)), 0) + rng.normal(0, 0.4, (N, P, 3)), L)
    wP = inputs.omega_P(P, BETA)
    V, F = oracle.long_double.fast_pimdb(pos, 1.0, wP, BETA, box=L)
    V, F = float(V), np.asarray(F, np.float64)
    for prec, (tv, tf) in TOL.items():
        eng = ExchangeEnergy(N, P, 1.0, wP, BETA, precision=prec, box=L, recompute=True)
        Vg, Fg = eng.forces(torch.from_numpy(pos).cuda())
        eng.sync()
        eng.close()
        assert abs(float(Vg) - V) <= tv * max(abs(V), 1.0 / BETA), prec
        assert np.linalg.norm(Fg.cpu().numpy() - F) <= tf * np.linalg.norm(F), prec
