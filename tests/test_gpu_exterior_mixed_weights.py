"""Weights of the mixed exterior forces: with coordinates on a grid of 2^-6 the
float32 differences, squares and spring energies are exact, so that what is left
is the weights' cut to float32 pairs and the pairs' products and sums.

Those round to nearest, so over many terms their errors average out; a cut that
truncates shows as a common shrinking of all weights.  For six particles a sum has
at most six terms: each within 2^-47 (weight) + 2^-47 (its product) + 2^-45 (sums of
at most eight low parts of 2^-23, each rounded at 2^-24 of it), below 2^-44 in all.
The mean over the 18,432 sums of 512 systems, a standard error of 2^-44 / 135 at the
most, stays within 2^-48; two factors cut at 2^-46 shrink it by 2^-46 on average.
"""
import numpy as np
import pytest
import torch

import oracle
from paper_2305_18025_gb300.exchange import BatchedExchangeEnergy, ExchangeEnergy

pytestmark = pytest.mark.gpu
N, P, R, WP, BETA = 6, 2, 512, 2.0, 0.25  # k = 4


def grid(N, seed):
    rng = np.random.default_rng(seed)
    c = np.cumsum(rng.integers(-40, 41, (N, 1, 3)), 0)
    return (c + rng.integers(-30, 31, (N, P, 3))) / 64.0


def sums(pos):
    """k times the probability-weighted sums of differences (bead P, bead 1), long double."""
    F, M = oracle.long_double.fast_pimdb(pos, 1.0, WP, BETA, full=True)[1::3]
    r = pos.astype(np.longdouble)
    pr = np.tril(np.asarray(M, np.longdouble))
    d = r[:, None, -1] - r[None, :, 0]
    t = pr[..., None] * d * 4
    return np.asarray(F, np.longdouble), t.sum(1), t.sum(0)


def shrink(got, F, rows, cols):
    """(sum of errors along the sums, sum of the sums): bead P's force holds -rows, bead 1's +cols."""
    err = got.astype(np.longdouble) - F
    along = -(err[:, -1] * np.sign(rows)).sum() + (err[:, 0] * np.sign(cols)).sum()
    return along, np.abs(rows).sum() + np.abs(cols).sum()


def test_mean_error_in_a_batch():
    ps = [grid(N, s) for s in range(R)]
    eng = BatchedExchangeEnergy([N] * R, [P] * R, 1.0, [WP] * R, [BETA] * R, precision="mixed")
    _, Fg = eng.forces(eng.pack([torch.from_numpy(p) for p in ps]))
    eng.sync()
    parts = [shrink(g.cpu().numpy(), *sums(p)) for g, p in zip(eng.unpack(Fg), ps)]
    eng.close()
    mean = float(sum(a for a, _ in parts) / sum(b for _, b in parts))
    assert abs(mean) <= 2.0 ** -48, mean * 2.0 ** 48


@pytest.mark.parametrize("recompute", [False, True])
def test_mean_error_of_a_long_system(recompute):
    n = 600
    pos = grid(n, 3)
    eng = ExchangeEnergy(n, P, 1.0, WP, BETA, precision="mixed", recompute=recompute)
    _, Fg = eng.forces(torch.from_numpy(pos).cuda())
    eng.sync()
    a, b = shrink(Fg.cpu().numpy(), *sums(pos))
    eng.close()
    # 3,600 sums; a row's terms are at most 600, a warp's 64: 2^-41 a sum, averaged over 60
    assert abs(float(a / b)) <= 2.0 ** -47, float(a / b) * 2.0 ** 48
