"""Running sums with infinite and NaN terms: as plain sums, infinite or NaN from that
term on."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mrc():
    from paper_2605_30379_gb300 import build
    build.build()
    from paper_2605_30379_gb300 import mrc as m
    m.load()
    return m


@pytest.mark.parametrize("at", [0, 255, 256, 700, 1499])
@pytest.mark.parametrize("bad", [np.inf, -np.inf, np.nan])
def test_visits(mrc, at, bad):
    """Chunks of 256 rows: the term in the first, at the seams, inside, in the last."""
    psi = np.random.default_rng(at).random((1500, 3, 3))
    psi[at, 1, 1] = bad
    v = mrc.renewal_visits(torch.from_numpy(psi).cuda(), torch.ones(3, dtype=torch.float64), [0, 1, 2]).cpu().numpy()
    assert np.isfinite(v[:at]).all()
    ref = np.cumsum(psi.sum(axis=(1, 2)))
    assert np.array_equal(v[at:], ref[at:], equal_nan=True)


def test_opposite_infinities_and_overflow(mrc):
    psi = np.zeros((600, 2, 2))
    psi[10, 0, 0], psi[300, 1, 1] = np.inf, -np.inf
    one = torch.ones(2, dtype=torch.float64)
    v = mrc.renewal_visits(torch.from_numpy(psi).cuda(), one, [0, 1]).cpu().numpy()
    assert (v[10:300] == np.inf).all() and np.isnan(v[300:]).all()
    psi[:] = 0.0
    psi[100:, 0, 0] = 1e308
    v = mrc.renewal_visits(torch.from_numpy(psi).cuda(), one, [0, 1]).cpu().numpy()
    assert v[100] == 1e308 and (v[101:] == np.inf).all()


def test_first_entrance_and_survival(mrc):
    """An infinite entrance kernel makes F infinite and S = 1 - F minus infinity (their
    convolution with the inverse is NaN from the transform on; the sums keep it)."""
    q = np.zeros((40, 2, 2))
    q[1, 0, 0], q[2, 0, 1] = 0.5, 0.5
    g, F, S = mrc.first_entrance(torch.from_numpy(q).cuda(), [1], torch.ones(1, dtype=torch.float64))
    assert torch.isfinite(F).all() and torch.isfinite(S).all()
    q[2, 0, 1] = np.inf
    g, F, S = mrc.first_entrance(torch.from_numpy(q).cuda(), [1], torch.ones(1, dtype=torch.float64))
    assert not torch.isfinite(F[2:]).any() and not torch.isfinite(S[2:]).any()
