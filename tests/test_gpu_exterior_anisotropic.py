"""Exterior-bead forces of flat systems: one axis 2^-30 of the others, each
component relative to its own largest force, with stored and recomputed pair
factors and in a replica batch, against the long-double oracle.

Tolerance (float64): the probabilities carry the recursions' error, within N 2^-51
in the worst case; a component's sum rounds at 2^-53 of its own terms.  At
N = 300: 300 (2^-51 + 2^-53) < 2^-42; asserted 1e-12 of the component's largest force.
"""
import numpy as np
import pytest
import torch

import oracle
from paper_2305_18025_gb300 import inputs
from paper_2305_18025_gb300.exchange import BatchedExchangeEnergy, ExchangeEnergy

pytestmark = pytest.mark.gpu
P, BETA = 3, 1.3


def system(N, axis):
    pos = inputs.clustered_chain_positions(N, P, seed=N)
    pos[..., axis] *= 2.0 ** -30
    F = oracle.long_double.fast_pimdb(pos, 1.0, inputs.omega_P(P, BETA), BETA)[1]
    return pos, np.asarray(F, np.float64)


def check(got, want):
    for c in range(3):
        assert np.abs(got[..., c] - want[..., c]).max() <= 1e-12 * np.abs(want[..., c]).max(), c


@pytest.mark.parametrize("N,axis", [(5, 2), (70, 0), (130, 1), (300, 2)])
@pytest.mark.parametrize("recompute", [False, True])
def test_each_component_to_its_own_size(N, axis, recompute):
    pos, F = system(N, axis)
    eng = ExchangeEnergy(N, P, 1.0, inputs.omega_P(P, BETA), BETA, recompute=recompute)
    _, Fg = eng.forces(torch.from_numpy(pos).cuda())
    eng.sync()
    check(Fg.cpu().numpy(), F)
    eng.close()


def test_each_component_to_its_own_size_in_a_batch():
    systems = [system(N, axis) for N, axis in ((70, 0), (33, 2), (130, 1))]
    n, w = [len(p) for p, _ in systems], inputs.omega_P(P, BETA)
    eng = BatchedExchangeEnergy(n, [P] * 3, 1.0, [w] * 3, [BETA] * 3)
    x = eng.pack([torch.from_numpy(p) for p, _ in systems])
    _, Fg = eng.forces(x)
    eng.sync()
    for got, (_, want) in zip(eng.unpack(Fg), systems):
        check(got.cpu().numpy(), want)
    eng.close()
