"""FP64 products of graded matrices: entries far below the largest of their row
or column keep the accuracy of floating FP64 sums."""
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


def birth_death(d, N, p=0.1):
    """Up with probability p, else down; geometric sojourns of mean 2.5."""
    k = np.arange(N)
    f = np.where(k > 0, 0.4 * 0.6 ** (k - 1.0), 0.0)
    q = np.zeros((N, d, d))
    for i in range(d):
        up = 1.0 if i == 0 else (0.0 if i == d - 1 else p)
        if up > 0.0:
            q[:, i, i + 1] = up * f
        if up < 1.0:
            q[:, i, i - 1] = (1.0 - up) * f
    return q


def entry_error(x, ref):
    """Largest error of an entry's series against that entry's largest value."""
    scale, err = np.abs(ref).max(axis=0), np.abs(x - ref).max(axis=0)
    assert (err[scale == 0.0] == 0.0).all()
    return (err[scale > 0.0] / scale[scale > 0.0]).max()


# The oracle's direct sums of nonnegative terms are accurate entry by entry; 2^-44
# per product of an entry 2^-10 to 2^-14 below its bounds, some ten to twenty
# products: 1e-12.
TOL = 1e-12


@pytest.mark.parametrize("d,N", [(4, 512), (20, 512), (28, 300), (40, 96), (40, 512), (64, 200)])
def test_birth_death_chain(mrc, d, N):
    """psi(i, j) falls by about a factor of ten per state; the entrance into the
    last state from the first has probabilities down to 1e-58."""
    q = birth_death(d, N)
    A = synth.identity_minus(q)
    psi = mrc.inverse(dev(A), prec="fp64").cpu().numpy()
    assert entry_error(psi, oracle.inverse_left(A)) <= TOL
    alpha = np.zeros(d - 1)
    alpha[0] = 1.0
    g, F, _ = mrc.first_entrance(dev(q), [d - 1], torch.tensor(alpha), prec="fp64")
    rg, rF, _ = oracle.first_entrance(q, [d - 1], alpha)
    assert entry_error(g.cpu().numpy(), rg) <= TOL
    assert abs(F[-1].item() / rF[-1] - 1.0) <= TOL


@pytest.mark.parametrize("d", [3, 20, 40])
@pytest.mark.parametrize("eps", [1e-6, 1e-10, 1e-14, 1e-20])
def test_rarely_reached_state(mrc, d, eps):
    rng = np.random.default_rng(d)
    P = rng.dirichlet(np.ones(d), size=d)
    P[:, d - 1] *= eps
    P /= P.sum(axis=1, keepdims=True)
    k = np.arange(300)
    A = synth.identity_minus(np.where(k > 0, 0.2 * 0.8 ** (k - 1.0), 0.0)[:, None, None] * P)
    psi = mrc.inverse(dev(A), prec="fp64").cpu().numpy()
    assert entry_error(psi, oracle.inverse_left(A)) <= TOL


@pytest.mark.parametrize("d", [4, 20, 31, 40, 64])
@pytest.mark.parametrize("span", [8, 30, 200])
def test_inner_scales(mrc, d, span):
    """Columns of A by 2^k and rows of B by 2^-k: every term of A * B, and so
    Prop 2.1's bound, stays what it was."""
    rng = np.random.default_rng(10 * d + span)
    N = 50
    A, B = rng.standard_normal((N, d, d)), rng.standard_normal((N, d, d))
    k = rng.integers(-span, span + 1, d)
    ref, _ = oracle.residuals(A, B)
    got = mrc.residual(dev(np.ldexp(A, k[None, None, :])), dev(np.ldexp(B, -k[None, :, None])), sides=1,
                       prec="fp64")[0].cpu().numpy()
    mrc.sync_status()
    L, u = 128, 2.0 ** -53
    sig, gam = 7 * u * np.log2(L), np.sqrt(2.0) * (d + 2) * u
    beta = 2 * sig + sig ** 2 + gam * (1 + sig) ** 2
    bound = np.sqrt(L) * np.sqrt((A ** 2).sum()) * np.sqrt((B ** 2).sum()) * (beta + sig * (1 + beta))
    assert np.sqrt(((got - ref) ** 2).sum()) <= bound


@pytest.mark.parametrize("d", [2, 6, 24, 40, 64])
def test_reducible_kernel(mrc, d):
    """States that never lead back: those entries of psi stay exactly zero, the
    others as accurate as ever."""
    rng = np.random.default_rng(d)
    P = rng.dirichlet(np.ones(d), size=d)
    P[d // 2:, :d // 2] = 0.0
    P /= P.sum(axis=1, keepdims=True)
    k = np.arange(200)
    A = synth.identity_minus(np.where(k > 0, 0.2 * 0.8 ** (k - 1.0), 0.0)[:, None, None] * P)
    psi = mrc.inverse(dev(A), prec="fp64").cpu().numpy()
    assert (psi[:, d // 2:, :d // 2] == 0.0).all()
    assert entry_error(psi, oracle.inverse_left(A)) <= TOL


def test_graded_models_in_a_batch(mrc):
    """One wave of graded and ordinary models, of the fixed-point and the digit
    products."""
    As = []
    for d, N in [(4, 300), (20, 129), (33, 200), (40, 96), (48, 200), (24, 64)]:
        As.append(synth.identity_minus(birth_death(d, N)))
        As.append(synth.identity_minus(synth.weibull_model(d, N, seed=d)[0]))
    outs = mrc.inverse_batched([dev(a) for a in As], prec="fp64")
    for a, x in zip(As, outs):
        ref = oracle.inverse_left(a)
        x = x.cpu().numpy()
        assert np.abs(x - ref).max() <= 1e-12
        if (a[:, 0, -1] == 0.0).all():  # the chains
            assert entry_error(x, ref) <= TOL


def test_tensor_core_row_and_column_scales(mrc):
    """The digit product's range (d >= 33): rows of A and columns of B by powers of
    two far apart scale the product exactly."""
    rng = np.random.default_rng(8)
    d, N = 40, 50
    A, B = rng.standard_normal((N, d, d)), rng.standard_normal((N, d, d))
    r, c = rng.integers(-200, 201, d), rng.integers(-200, 201, d)
    one = mrc.residual(dev(A), dev(B), sides=1, prec="fp64")[0].cpu().numpy()
    two = mrc.residual(dev(np.ldexp(A, r[None, :, None])), dev(np.ldexp(B, c[None, None, :])), sides=1,
                       prec="fp64")[0].cpu().numpy()
    two = np.ldexp(np.ldexp(two, -r[None, :, None]), -c[None, None, :])
    assert np.array_equal(one[1:], two[1:])  # (row 0 holds the identity)


@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
@pytest.mark.parametrize("d", [40, 64])
def test_tensor_core_non_finite(mrc, d, bad):
    rng = np.random.default_rng(9)
    A, B = rng.standard_normal((40, d, d)), rng.standard_normal((40, d, d))
    ref = mrc.residual(dev(A), dev(B), sides=1, prec="fp64")[0]
    B[3, 5, 7] = bad
    got = mrc.residual(dev(A), dev(B), sides=1, prec="fp64")[0]
    assert not torch.isfinite(got[:, :, 7]).any()
    keep = [j for j in range(d) if j != 7]
    assert torch.equal(got[:, :, keep], ref[:, :, keep])
    A[5, 33, 2], B[3, 5, 7] = bad, 0.5
    ref = mrc.residual(dev(np.where(np.isfinite(A), A, 0.0)), dev(B), sides=1, prec="fp64")[0]
    got = mrc.residual(dev(A), dev(B), sides=1, prec="fp64")[0]
    assert not torch.isfinite(got[:, 33]).any()
    keep = [i for i in range(d) if i != 33]
    assert torch.equal(got[:, keep], ref[:, keep])
