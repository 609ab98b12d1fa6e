"""Rounding of the recursions: coincident particles have no springs, every pair
factor is 1 and V_B is 0 but for the rounding of the coefficients 1 / l to float64,
which the same recursion in long double carries too.

Tolerance: an entry of the recursion adds at most 72 products, each cut at 2^-59 of
the largest, half of that on average and always downwards: 2^-54 an entry.  y_l
carries its own error and the mean of the earlier ones, so ln y_N at most
(1 + ln N) 2^-54; the cut of y_N to 53 bits and its logarithm add 4 2^-53.
"""
import numpy as np
import pytest
import torch

from paper_2305_18025_gb300 import inputs
from paper_2305_18025_gb300.exchange import BatchedExchangeEnergy, ExchangeEnergy

pytestmark = pytest.mark.gpu


def exact(N):
    """-ln y_N with y_l = c_l sum_{w<l} y_w, c_l = 1 / l rounded to float64."""
    total, y = np.longdouble(1), np.longdouble(1)
    for l in range(1, N + 1):
        y = np.longdouble(1.0 / l) * total
        total += y
    return float(-np.log(y))


def near(V, N):
    return abs(V - exact(N)) <= ((1 + np.log(N)) / 2 + 4) * 2.0 ** -53


@pytest.mark.parametrize("N", [64, 128, 129, 1024, 1601, 2048, 4096])
@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("recompute", [False, True])
def test_coincident_particles(N, prec, recompute):
    eng = ExchangeEnergy(N, 2, 1.0, 2.0, 1.0, precision=prec, recompute=recompute)
    V, _ = eng.forces(torch.from_numpy(inputs.coincident_positions(N, 2)).cuda())
    eng.sync()
    eng.close()
    assert near(float(V), N), float(V) * 2.0 ** 53


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
def test_coincident_replicas(prec):
    n = [33, 512, 1500]
    eng = BatchedExchangeEnergy(n, [2] * 3, 1.0, [2.0] * 3, [1.0] * 3, precision=prec)
    V, _ = eng.forces(eng.pack([torch.from_numpy(inputs.coincident_positions(k, 2)) for k in n]))
    eng.sync()
    eng.close()
    for v, k in zip(V.tolist(), n):
        assert near(v, k), (k, v * 2.0 ** 53)
