"""The FP64 path's fixed-point transforms and digit products at the sizes and
values where they can go wrong, against the oracle's direct sums."""
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


def product_bound(A, B, u=2.0 ** -53):
    """Prop 2.1's forward-error bound of the FFT product (the constants of
    test_fft_product_within_prop_2_1_bound)."""
    N, d = A.shape[0], A.shape[1]
    L = 2 << max(0, (N - 1).bit_length())
    sig, gam = 7 * u * np.log2(L), np.sqrt(2.0) * (d + 2) * u
    beta = 2 * sig + sig ** 2 + gam * (1 + sig) ** 2
    norm = lambda X: np.sqrt((X ** 2).sum())
    return np.sqrt(L) * norm(A) * norm(B) * (beta + sig * (1 + beta))


def integers(rng, N, d):
    return rng.integers(-8, 9, size=(N, d, d)).astype(np.float64)


@pytest.mark.parametrize("d", [1, 3])
@pytest.mark.parametrize("N", [1, 2, 3, 4, 5, 8, 9, 16, 17, 33, 65, 129, 257, 513, 1024, 1025, 2049, 4097])
def test_transform_sizes(mrc, N, d):
    """One transform length per power of two up to two passes, ragged row
    counts, E = 1 and 9 (partial entry chunks): rho = e0 - A * B on small
    integers, whose direct sums are exact, within 1 % of Prop 2.1's bound
    (N >= 2; a few roundings of the entries at N = 1)."""
    rng = np.random.default_rng(1000 * d + N)
    A, B = integers(rng, N, d), integers(rng, N, d)
    ref, _ = oracle.residuals(A, B)
    got = mrc.residual(dev(A), dev(B), sides=1, prec="fp64")[0].cpu().numpy()
    assert np.sqrt(((got - ref) ** 2).sum()) <= max(1e-2, 0.2 / N) * product_bound(A, B)


@pytest.mark.parametrize("e", [300, -300, 900])
def test_power_of_two_scaling_is_exact(mrc, e):
    """The alignment follows each column's exponent: scaling A by 2^e and B by
    2^-e changes no bit of their product."""
    rng = np.random.default_rng(5)
    A, B = rng.standard_normal((300, 3, 3)), rng.standard_normal((300, 3, 3))
    one = mrc.residual(dev(A), dev(B), sides=1, prec="fp64")[0]
    two = mrc.residual(dev(np.ldexp(A, e)), dev(np.ldexp(B, -e)), sides=1, prec="fp64")[0]
    assert torch.equal(one, two)


@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
def test_non_finite_values_stay_in_their_row(mrc, bad):
    """A NaN or infinity in A(k)[1][2] reaches row 1 of A * B and no other row;
    nothing finite comes out of that row's product."""
    rng = np.random.default_rng(6)
    A, B = rng.standard_normal((40, 3, 3)), rng.standard_normal((40, 3, 3))
    ref = mrc.residual(dev(A), dev(B), sides=1, prec="fp64")[0]
    A[7, 1, 2] = bad
    got = mrc.residual(dev(A), dev(B), sides=1, prec="fp64")[0]
    assert not torch.isfinite(got[:, 1]).any()
    assert torch.equal(got[:, [0, 2]], ref[:, [0, 2]])


@pytest.mark.parametrize("d,N,seed", [(3, 2048, 0), (16, 2049, 1), (40, 700, 2)])
def test_long_tails_and_spikes(mrc, d, N, seed):
    """A = e0 - q: unit spikes beside entries of 1e-3 that fall off to nothing;
    the inverse keeps the FP64 tolerance."""
    q, _ = synth.weibull_model(d, N, seed=seed)
    A = synth.identity_minus(q)
    psi = mrc.inverse(dev(A), prec="fp64").cpu().numpy()
    assert np.abs(psi - oracle.inverse_left(A)).max() <= 1e-12


@pytest.mark.parametrize("N", [1, 2, 3, 40])
@pytest.mark.parametrize("d", [15, 16, 17, 31, 32, 33, 48, 49, 63, 64, 65])
def test_digit_product_sizes(mrc, d, N):
    """The FP64 digit product (17 <= d <= 64: two to four K chunks of 16, full
    and ragged) and the sizes just outside: M = 1 (the self-paired frequency
    alone), 2, 4 and 64 points, integers with exact direct sums."""
    rng = np.random.default_rng(100 * d + N)
    A, B = integers(rng, N, d), integers(rng, N, d)
    ref, _ = oracle.residuals(A, B)
    got = mrc.residual(dev(A), dev(B), sides=1, prec="fp64")[0].cpu().numpy()
    mrc.sync_status()
    assert np.sqrt(((got - ref) ** 2).sum()) <= max(1e-2, 0.2 / N) * product_bound(A, B)


def test_digit_product_row_and_column_scales(mrc):
    """Rows of A and columns of B scaled by powers of two far apart: row i and
    column j of the product scale exactly (rows and columns are aligned each by
    itself)."""
    rng = np.random.default_rng(8)
    d, N = 20, 50
    A, B = rng.standard_normal((N, d, d)), rng.standard_normal((N, d, d))
    r, c = rng.integers(-200, 201, d), rng.integers(-200, 201, d)
    A[0] += 3 * np.eye(d)
    one = -mrc.residual(dev(A), dev(B), sides=1, prec="fp64")[0].cpu().numpy()
    one[0] += np.eye(d)
    two = -mrc.residual(dev(np.ldexp(A, r[None, :, None])), dev(np.ldexp(B, c[None, None, :])), sides=1,
                        prec="fp64")[0].cpu().numpy()
    two = np.ldexp(two, -r[None, :, None])
    two = np.ldexp(two, -c[None, None, :])
    assert np.array_equal(one[1:], two[1:])


@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_digit_product_non_finite(mrc, bad):
    rng = np.random.default_rng(9)
    A, B = rng.standard_normal((40, 20, 20)), rng.standard_normal((40, 20, 20))
    ref = mrc.residual(dev(A), dev(B), sides=1, prec="fp64")[0]
    B[3, 5, 7] = bad
    got = mrc.residual(dev(A), dev(B), sides=1, prec="fp64")[0]
    assert not torch.isfinite(got[:, :, 7]).any()
    keep = [j for j in range(20) if j != 7]
    assert torch.equal(got[:, :, keep], ref[:, :, keep])


@pytest.mark.parametrize("d,c", [(1, 1), (2, 7), (5, 3), (24, 3), (40, 2), (56, 1), (78, 1), (80, 5), (20, 130)])
def test_rectangular_products(mrc, d, c):
    """V = psi * r with c columns: the fixed-point product (several pairs per
    CTA, ragged last CTA, one pair of up to 200 KB) and, for spectra that do
    not fit, the tiles (d = 80); integers, within 1 % of Prop 2.1's bound."""
    rng = np.random.default_rng(10 * d + c)
    N = 70
    X = rng.integers(-8, 9, size=(N, d, d)).astype(np.float64)
    r = rng.integers(-8, 9, size=(N, d, c)).astype(np.float64)
    V = mrc.reward(dev(X), dev(r), prec="fp64").cpu().numpy()
    ref = oracle.convolve(X, r)
    assert np.sqrt(((V - ref) ** 2).sum()) <= 1e-2 * product_bound(X, r)


@pytest.mark.parametrize("d,N", [(2, 1), (3, 255), (31, 256), (32, 257), (33, 700), (7, 70000)])
def test_functionals_sizes(mrc, d, N):
    """Running sums over one, full, ragged and many chunks and 1 to 33 columns,
    weighted sums of matrices narrower and wider than a warp, and the diagonal
    product: visits, occupation and transition against numpy sums (transition:
    rows add up to one for psi = the inverse, checked on the horizon the
    oracle reaches)."""
    rng = np.random.default_rng(d)
    psi, alpha = rng.uniform(0, 1, (N, d, d)), rng.uniform(0, 1, d)
    B = sorted(rng.choice(d, max(1, d // 2), replace=False).tolist())
    occ = np.einsum("i,kij->k", alpha, psi[:, :, B])
    got = mrc.occupation(dev(psi), torch.tensor(alpha), B).cpu().numpy()
    assert np.abs(got - occ).max() <= 1e-15 * d * d
    vis = mrc.renewal_visits(dev(psi), torch.tensor(alpha), B).cpu().numpy()
    ref = np.cumsum(occ.astype(np.longdouble)).astype(float)
    assert np.abs(vis - ref).max() <= 1e-15 * (d * d + np.log2(N + 1)) * max(1.0, ref.max())
    n = min(N, 1500)
    q, _ = synth.weibull_model(d, n, seed=d)
    x = oracle.inverse_left(synth.identity_minus(q))
    P = mrc.transition(dev(x), dev(q), prec="fp64").cpu().numpy()
    assert np.abs(P - oracle.transition(x, q)).max() <= 1e-13
    assert np.abs(P.sum(axis=2) - 1.0).max() <= 1e-12


def test_diagonal_product_non_finite(mrc):
    q, _ = synth.weibull_model(5, 40, seed=1)
    psi = torch.rand(40, 5, 5, dtype=torch.float64, device="cuda")
    ref = mrc.transition(psi, dev(q))
    psi[3, 2, 1] = float("inf")
    got = mrc.transition(psi, dev(q))
    assert not torch.isfinite(got[:, 2, 1]).any()
    got[:, 2, 1] = ref[:, 2, 1]
    assert torch.equal(got, ref)


@pytest.mark.parametrize("d", [1, 2, 4, 10, 16, 25, 26, 32, 33, 47, 48, 64, 100, 256])
def test_seed_sizes(mrc, d):
    """The start of the doubling on one cluster: A(0) with a zero diagonal (every
    pivot from another row) and dense signed coefficients, horizons below, at
    and beyond the direct levels (256 coefficients at d <= 4 down to 2 for
    d > 32), rows spread evenly and unevenly over the 16 CTAs."""
    rng = np.random.default_rng(d)
    for N in ([1, 2, 3, 7, 255, 256, 300] if d <= 4 else [1, 2, 5, 33] if d <= 64 else [1, 3]):
        A = rng.standard_normal((N, d, d)) * (0.5 ** np.arange(N))[:, None, None] * 0.2 / d
        A[0] += np.roll(np.diag(2.0 + np.arange(d)), 1, axis=1)
        ref = oracle.inverse_left(A)
        psi = mrc.inverse(dev(A), prec="fp64", report=True)[0].cpu().numpy()
        assert np.abs(psi - ref).max() <= 1e-12 * max(1.0, np.abs(ref).max())


@pytest.mark.parametrize("d", [3, 32, 33, 100, 512])
def test_seed_singular(mrc, d):
    rng = np.random.default_rng(d)
    A = np.zeros((4, d, d))
    A[0] = rng.standard_normal((d, d))
    A[0, :, d - 1] = 0.0
    with pytest.raises(mrc.MrcError) as ei:
        mrc.inverse(dev(A), prec="fp64", report=True)
    assert ei.value.status == 2
    assert torch.isnan(mrc.inverse(dev(A), prec="fp64")[0]).all()
    with pytest.raises(mrc.MrcError):
        mrc.sync_status()
    eye = torch.eye(d, dtype=torch.float64, device="cuda")[None]
    assert torch.equal(mrc.inverse(eye, report=True)[0], eye)


@pytest.mark.parametrize("N", [5, 2048, 32768])
def test_running_sums_in_small_scratch(mrc, N, monkeypatch):
    """A workspace cap of 256 B makes the running sums' chunks longer: the same
    sums to a rounding of each (they are kept as unevaluated pairs)."""
    rng = np.random.default_rng(N)
    psi, alpha = dev(rng.random((N, 3, 3))), dev(rng.random(3))
    ref = mrc.renewal_visits(psi, alpha, [0, 2])
    ctx = mrc.create_context(max_workspace_bytes=256)
    try:
        monkeypatch.setattr(mrc, "context", lambda device=None: ctx)
        got = mrc.renewal_visits(psi, alpha, [0, 2])
        torch.cuda.synchronize()
    finally:
        monkeypatch.undo()
        mrc.destroy_context(ctx)
    assert ((got - ref).abs() <= 2.0 ** -52 * ref.abs()).all()
