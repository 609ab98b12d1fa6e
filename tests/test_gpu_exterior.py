"""Exterior-bead forces by tile items, at the edges of tiles and of the launch
shapes (one, two, four and eight CTAs an item), with stored and recomputed
pair factors, against the long-double oracle.

Tolerances.  FP64: the recursions truncate below 2^-51 relative a row (a few
2^-56 terms each), so y, mu and 1/(N y_N) are within N 2^-51 of their values in
the worst case, 2^-40 at N = 2049; the sums add 2^-57 a term.  Asserted: 1e-12.
Mixed: float32 bead differences (2^-24 of coordinates of order 1, against
differences of order 0.1) enter each force once: 1e-6 in the 2-norm.
"""
import numpy as np
import pytest
import torch

import oracle
from paper_2305_18025_gb300 import inputs
from paper_2305_18025_gb300.bpimd import BpimdError
from paper_2305_18025_gb300.exchange import ExchangeEnergy

pytestmark = pytest.mark.gpu

SIZES = [1, 2, 31, 32, 33, 63, 64, 65, 97, 128, 129, 257, 1023, 1025, 2047, 2049]


@pytest.mark.parametrize("N", SIZES)
def test_exterior_forces_at_tile_and_launch_edges(N):
    P, beta = 3, 1.3
    wP = inputs.omega_P(P, beta)
    pos = inputs.clustered_chain_positions(N, P, seed=40 + N)
    V, F = oracle.long_double.fast_pimdb(pos, 1.0, wP, beta)
    norm = np.linalg.norm(F)
    x = torch.from_numpy(pos).cuda()
    for prec, tol in (("fp64", 1e-12), ("mixed", 1e-6), ("mixed32", 1e-5)):
        for recompute in (False, True):
            eng = ExchangeEnergy(N, P, 1.0, wP, beta, precision=prec, recompute=recompute)
            Vg, Fg = eng.forces(x)
            eng.sync()
            assert abs(float(Vg) - V) <= max(tol, 1e-12) * max(abs(V), 1.0 / beta), (prec, recompute)
            assert np.linalg.norm(Fg.cpu().numpy() - F) <= tol * norm, (prec, recompute)
            eng.close()


@pytest.mark.parametrize("prec", ["fp64", "mixed", "mixed32"])
@pytest.mark.parametrize("recompute", [False, True])
def test_a_non_finite_endpoint_reaches_its_forces_and_the_status(prec, recompute):
    N, P, beta = 70, 3, 1.0
    pos = inputs.clustered_chain_positions(N, P, seed=7)
    pos[33, P - 1, 1] = np.nan
    eng = ExchangeEnergy(N, P, 1.0, inputs.omega_P(P, beta), beta, precision=prec, recompute=recompute)
    _, F = eng.forces(torch.from_numpy(pos).cuda())
    assert not torch.isfinite(F[33, P - 1, 1])
    with pytest.raises(BpimdError):
        eng.sync()
    eng.close()
