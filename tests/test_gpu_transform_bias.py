"""The FP64 transforms round symmetrically: the result for -x is minus the result for x
up to roundings of either sign.  (A direction would add up in the zero frequency,
which the inverse of e0 - q amplifies by the horizon.)"""
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


@pytest.mark.parametrize("N", [128, 256, 512, 1024, 2048, 4096])
def test_sum_over_time_is_odd(mrc, N):
    """C(A) + C(-A) for C(A) = A * e0, summed over time, for 4 x 24^2 columns of one minus a
    decaying series of sum about 0.6: the mean over the columns.  Each of the two
    transforms rounds the zero frequency, about 0.4, once to FP64: errors of at most
    2^-54 whose signs differ from column to column; the mean of so many stays
    below five times 2^-53 over the square root of their number."""
    rng = np.random.default_rng(N)
    d, asym = 24, []
    e0 = torch.zeros((N, d, d), dtype=torch.float64, device="cuda")
    e0[0] = torch.eye(d, dtype=torch.float64)
    for _ in range(4):
        lam, w = rng.uniform(3.0, 12.0, (d, d)), rng.uniform(0.4, 0.8, (d, d))
        k = np.arange(N)[:, None, None]
        A = -w * np.exp(-(k - 1.0) / lam) * (1.0 - np.exp(-1.0 / lam))
        A[0] = 1.0
        A = torch.from_numpy(A).cuda()
        # e0 - A * e0 and e0 + A * e0
        C = [mrc.residual(x, e0, sides=1, prec="fp64")[0].cpu().numpy().astype(np.longdouble) for x in (A, -A)]
        s = C[0] + C[1]
        s[0] -= 2 * np.eye(d)
        asym.append(s.sum(axis=0) / 2)
    assert abs(float(np.mean(asym))) <= 5 * 2.0 ** -53 / np.sqrt(4 * d * d)
