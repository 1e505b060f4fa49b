"""FP64 calls near the ends of the number range: scaling an input by a power of two
scales the result, down to where it becomes subnormal."""
import numpy as np
import pytest
import torch

import oracle
from paper_2605_30379_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mrc():
    from paper_2605_30379_gb300 import build
    build.build()
    from paper_2605_30379_gb300 import mrc as m
    m.load()
    return m


def dev(x):
    return torch.from_numpy(np.ascontiguousarray(x)).to("cuda")


def tolerance(top):
    """1e-12 (the FP64 tolerance) and four spacings of the subnormals against results of
    at most 2^top."""
    return 1e-12 + 4.0 * 2.0 ** (-1074 - top)


@pytest.mark.parametrize("d,N", [(1, 300), (3, 1500), (12, 700), (40, 200), (64, 70)])
@pytest.mark.parametrize("e", [940, 960, 990, 1005, -940, -960, -990, -1005])
def test_inverse_of_scaled_sequences(mrc, d, N, e):
    """(2^e A)^(-1) = 2^-e A^(-1): results of about 2^-e."""
    q, _ = synth.weibull_model(max(d, 2), N, seed=d)
    A = synth.identity_minus(q[:, :d, :d])
    ref = oracle.inverse_left(A)
    got = np.ldexp(mrc.inverse(dev(np.ldexp(A, e)), prec="fp64").cpu().numpy(), e)
    mrc.sync_status()
    assert np.abs(got - ref).max() <= tolerance(-e) * max(1.0, np.abs(ref).max())


@pytest.mark.parametrize("d,c", [(1, 1), (4, 2), (24, 3), (40, 40), (64, 64), (80, 5)])
@pytest.mark.parametrize("ex,ey", [(-1000, 0), (0, -1000), (-1030, 30), (-520, -500), (-1000, 900), (900, -1000),
                                   (-600, -600)])
def test_products_of_scaled_sequences(mrc, d, c, ex, ey):
    """psi * r with psi by 2^ex and r by 2^ey (both subnormal in part at -1030, the
    product below the range at -1200): fixed-point and digit products and tiles."""
    rng = np.random.default_rng(d + c)
    X, r = rng.random((70, d, d)), rng.random((70, d, c))
    ref = oracle.convolve(X, r)
    got = mrc.reward(dev(np.ldexp(X, ex)), dev(np.ldexp(r, ey)), prec="fp64").cpu().numpy()
    if ex + ey < -1100:
        assert (np.abs(got) <= 2.0 ** -1074 * 8).all()
        return
    # (entries of X and r below 2^-1022 were rounded to multiples of 2^-1074 going in)
    tol = tolerance(ex + ey) + 2.0 ** (-1073 - min(ex, 0)) + 2.0 ** (-1073 - min(ey, 0))
    assert np.abs(np.ldexp(got, -(ex + ey)) - ref).max() <= tol * ref.max()


@pytest.mark.parametrize("e", [-900, -960, -1000, 960])
def test_transition_of_scaled_sequences(mrc, e):
    """The diagonal product: P = psi * diag(survival) with psi by 2^e."""
    q, _ = synth.weibull_model(5, 300, seed=1)
    psi = oracle.inverse_left(synth.identity_minus(q))
    ref = mrc.transition(dev(psi), dev(q), prec="fp64").cpu().numpy()
    got = np.ldexp(mrc.transition(dev(np.ldexp(psi, e)), dev(q), prec="fp64").cpu().numpy(), -e)
    assert np.abs(got - ref).max() <= tolerance(e)
