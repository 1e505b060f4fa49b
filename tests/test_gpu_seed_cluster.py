"""Gauss-Jordan on clusters of 8 and 16 CTAs, with the rows in shared memory and (8
CTAs, d > 460) in device memory."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mrc():
    from paper_2605_30379_gb300 import build
    build.build()
    from paper_2605_30379_gb300 import mrc as m
    m.load()
    return m


def status(mrc, call, *args):
    """The status a call raises (no exception kept: its frames would hold device tensors
    until a later collection)."""
    try:
        call(*args)
    except mrc.MrcError as e:
        return e.status
    return 0


@pytest.mark.parametrize("cluster", [8, 16])
@pytest.mark.parametrize("d", [1, 3, 32, 33, 100, 457, 459, 460, 461, 500, 512])
def test_inverse(mrc, d, cluster):
    """Every pivot from another row; against the oracle's elimination, to a few
    roundings per column of entries of order one."""
    rng = np.random.default_rng(d)
    A = rng.standard_normal((d, d)) / d + np.roll(np.diag(1.0 + rng.random(d)), 1, axis=1)
    got = mrc.selftest_gauss_jordan(torch.from_numpy(A).cuda(), cluster).cpu().numpy()
    mrc.sync_status()
    assert np.abs(got - oracle.gauss_jordan(A)).max() <= 16 * d * 2.0 ** -53


@pytest.mark.parametrize("cluster", [8, 16])
@pytest.mark.parametrize("d", [5, 64, 512])
def test_singular(mrc, d, cluster):
    A = np.random.default_rng(d).standard_normal((d, d))
    A[:, d // 2] = 0.0
    assert torch.isnan(mrc.selftest_gauss_jordan(torch.from_numpy(A).cuda(), cluster)).all()
    assert status(mrc, mrc.sync_status) == 2


def test_arguments(mrc):
    A = torch.eye(4, dtype=torch.float64, device="cuda")
    assert status(mrc, mrc.selftest_gauss_jordan, A, 4) == 1
