"""A non-finite coordinate of an interior bead reaches, through the Gaussian pairs,
that component of every other particle's bead of the same index: interior beads of
different particles share nothing else.  Other components and beads stay finite.
"""
import numpy as np
import pytest
import torch

from paper_2305_18025_gb300 import inputs
from paper_2305_18025_gb300.bpimd import BpimdError
from paper_2305_18025_gb300.exchange import BatchedExchangeEnergy, RingPolymerMD

pytestmark = pytest.mark.gpu
N, P = 40, 6


def start(value):
    pos = np.random.default_rng(3).normal(0.0, 1.0, (N, P, 3))
    pos[7, 2, 1] = value
    return torch.from_numpy(pos).cuda()


def check(v):
    v = v.cpu().numpy()
    others = np.arange(N) != 7
    assert not np.isfinite(v[others, 2, 1]).any()
    assert np.isfinite(v[others, 2, 0]).all() and np.isfinite(v[others, 2, 2]).all()
    assert np.isfinite(v[others][:, 4]).all()


@pytest.mark.parametrize("value", [np.inf, np.nan])
def test_single_system(value):
    md = RingPolymerMD(N, P, 1.0, inputs.omega_P(P, 1.0), 1.0, dt=0.01, gamma=0.0, gaussian=(3.0, 0.5))
    x, v = start(value), torch.zeros((N, P, 3), dtype=torch.float64, device="cuda")
    with pytest.raises(BpimdError, match="non-finite"):
        md.step(x, v, 1)
    check(v)
    md.close()


@pytest.mark.parametrize("value", [np.inf, np.nan])
def test_replica(value):
    eng = BatchedExchangeEnergy([N, 5], [P, P], 1.0, [inputs.omega_P(P, 1.0)] * 2, [1.0] * 2,
                                md=dict(dt=0.01, gamma=0.0, gaussian=(3.0, 0.5)))
    x = eng.pack([start(value), torch.zeros((5, P, 3), dtype=torch.float64).cuda()])
    v = torch.zeros_like(x)
    with pytest.raises(BpimdError, match="non-finite"):
        eng.step(x, v, 1)
    a, b = eng.unpack(v)
    check(a)
    assert torch.isfinite(b).all()
    eng.close()
