"""Performance cases: the work a user of the library has it do, through the
Python entry points, over the sizes and options they are used with.

A case is a dict of plain values: "kind" says which entry points it calls,
"d" / "N" the matrix dimension and horizon, "prec" the precision option.

Inputs are seeded semi-Markov kernels of the shapes the configurations,
tests and benchmark use (discrete Weibull and shifted Gamma sojourns,
Lognormal sojourns under the endpoint mean-value rule, the exponential
four-state generator), evaluated on the GPU.  `exact` recomputes a case with
torch's FP64 FFTs and matrix products alone.
"""
import math

import numpy as np
import torch

from paper_2605_30379_gb300 import mrc

DEV = "cuda"
F64 = torch.float64


def listed():
    return [
        # One small model, the paper's 3-state example at its shortest horizon:
        # what an interactive session or a fitting loop calls again and again.
        {"name": "inverse_d3_N128_fp64", "kind": "inverse", "model": "gamma", "d": 3, "N": 128, "prec": "fp64"},
        # The same model at the longest horizon of the paper's timing table.
        {"name": "inverse_d3_N2048_fp64", "kind": "inverse", "model": "gamma", "d": 3, "N": 2048, "prec": "fp64"},
        # The default precision on the mid-size Weibull configuration.
        {"name": "inverse_d16_N8192_fp64", "kind": "inverse", "model": "weibull", "d": 16, "N": 8192, "prec": "fp64"},
        # The default precision at the dimension of the headline workload.
        {"name": "inverse_d64_N32768_fp64", "kind": "inverse", "model": "lognormal", "d": 64, "N": 32768,
         "prec": "fp64"},
        # The mixed path on a long-horizon Weibull model of moderate dimension.
        {"name": "inverse_d16_N65536_mixed", "kind": "inverse", "model": "weibull", "d": 16, "N": 65536,
         "prec": "mixed", "sweeps": 1},
        # A horizon and a dimension that are no round numbers.
        {"name": "inverse_d45_N20011_mixed", "kind": "inverse", "model": "weibull", "d": 45, "N": 20011,
         "prec": "mixed", "sweeps": 1},
        # Dense precision stress: large matrices, two refinement sweeps.
        {"name": "inverse_d256_N4096_mixed", "kind": "inverse", "model": "weibull", "d": 256, "N": 4096,
         "prec": "mixed", "sweeps": 2},
        # The headline workload of the benchmark.
        {"name": "inverse_d64_N262144_mixed", "kind": "inverse", "model": "lognormal", "d": 64, "N": 262144,
         "prec": "mixed", "sweeps": 1},
        # Many independent models of uneven sizes at once (a bootstrap or a
        # portfolio): d in 3..48, N in 2^10..2^14, half Weibull, half Lognormal.
        {"name": "batch_32_mixed", "kind": "batch", "n": 32, "dlo": 3, "dhi": 48, "lo": 10.0, "hi": 14.0,
         "prec": "mixed", "sweeps": 1},
        # Continuous time: the transition function of the four-state
        # exponential benchmark on its finest grid.
        {"name": "mre_d4_N32768_fp64", "kind": "mre", "model": "exponential", "d": 4, "N": 32768, "prec": "fp64"},
        # Reliability of a mid-size system: first entrance into the failed states.
        {"name": "entrance_d24_N10000_fp64", "kind": "entrance", "d": 24, "nD": 6, "N": 10000, "prec": "fp64"},
        # The functionals of a renewal sequence already in hand: transition
        # function, availability, expected visits, rewards.
        {"name": "functionals_d32_N16384_fp64", "kind": "functionals", "d": 32, "c": 2, "N": 16384, "prec": "fp64"},
    ]


# ---------------------------------------------------------------------------
# drawn cases

def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _load(d, N, prec):
    """Rough time of one inverse: transforms and products, FP64 dearer."""
    return float(N) * d * d * (5.0 * math.log2(2 * N) + 8.0 * d) * (6.0 if prec == "fp64" else 1.0)


_LOAD_MAX = 0.8 * _load(64, 262144, "mixed")


def draw(rng):
    kind = rng.choice(["inverse", "inverse", "inverse", "inverse", "batch", "mre", "entrance", "functionals"])
    prec = rng.choice(["fp64", "mixed"])
    if kind == "batch":
        return {"kind": kind, "n": rng.randint(4, 48), "dlo": 3, "dhi": rng.randint(8, 48), "lo": 10.0,
                "hi": round(rng.uniform(11.0, 14.0), 2), "prec": prec, "sweeps": 1}
    while True:
        if kind == "inverse":
            d, N = _log_int(rng, 3, 256), _log_int(rng, 128, 262144)
        elif kind == "mre":
            d, N = _log_int(rng, 3, 16), _log_int(rng, 1000, 65536)
        elif kind == "entrance":
            d, N = _log_int(rng, 3, 48), _log_int(rng, 128, 32768)
        else:
            d, N = _log_int(rng, 3, 64), _log_int(rng, 500, 32768)
        if _load(d, N, prec) <= _LOAD_MAX and N * d * d <= 1 << 28:
            break
    if kind == "inverse":
        return {"kind": kind, "model": rng.choice(["weibull", "lognormal"]), "d": d, "N": N, "prec": prec,
                "sweeps": 2 if d >= 128 and prec == "mixed" else 1}
    if kind == "mre":
        return {"kind": kind, "model": "lognormal", "d": d, "N": N, "prec": prec}
    if kind == "entrance":
        return {"kind": kind, "d": d, "nD": rng.randint(1, max(1, d // 3)), "N": N, "prec": prec}
    return {"kind": kind, "d": d, "c": rng.randint(1, 4), "N": N, "prec": prec}


# ---------------------------------------------------------------------------
# inputs

def _rng(seed, salt):
    return np.random.default_rng([int(seed), salt])


def _chain(g, d):
    """Embedded chain: zero diagonal, Dirichlet(1) rows."""
    P = g.gamma(1.0, size=(d, d))
    np.fill_diagonal(P, 0.0)
    return P / P.sum(axis=1, keepdims=True)


def _dev(x):
    return torch.from_numpy(np.ascontiguousarray(x)).to(DEV)


def _rows(N, d):
    """Row ranges of at most 2^24 entries."""
    step = max(1, (1 << 24) // (d * d))
    return [(s, min(N, s + step)) for s in range(0, N, step)]


def _weibull_q(g, d, N):
    """q(k) = P f(k), f(k) = P(k - 1 <= X < k) for Weibull X, q(0) = 0."""
    P, beta, lam = _dev(_chain(g, d)), _dev(g.uniform(0.8, 2.0, (d, d))), _dev(g.uniform(2.0, 20.0, (d, d)))
    q = torch.empty((N, d, d), dtype=F64, device=DEV)
    for s, e in _rows(N, d):
        k = torch.arange(s, e, dtype=F64, device=DEV)[:, None, None]
        hi = torch.exp(-torch.pow(torch.clamp(k - 1.0, min=0.0) / lam, beta))
        q[s:e] = P * (hi - torch.exp(-torch.pow(k / lam, beta)))
    q[0] = 0.0
    return q


def _gamma_q(g, N):
    """The paper's three-state kernel with shifted discrete Gamma sojourns,
    shapes and scales varied a little by the seed; q(0) = 0."""
    q = np.zeros((N, 3, 3))
    k = torch.arange(0, N, dtype=F64)
    for (i, j), (a, th, w) in {(0, 1): (1.8, 4.0, 1.0), (1, 0): (1.6, 5.0, 0.2), (1, 2): (2.2, 4.0, 0.8),
                               (2, 0): (1.9, 3.0, 1.0)}.items():
        a, th = a * g.uniform(0.9, 1.1), th * g.uniform(0.9, 1.1)
        cdf = torch.special.gammainc(torch.full_like(k, a), k / th).numpy()
        q[1:, i, j] = w * (cdf[1:] - cdf[:-1])
    return _dev(q)


def _lognormal_Q(g, d, n, h=0.05):
    """Q(m h) = P Phi((log mh - mu) / sigma), m = 0 .. n, as a function of a row range."""
    P, sig, mu = _dev(_chain(g, d)), _dev(g.uniform(1.0, 2.0, (d, d))), _dev(g.uniform(0.0, 3.0, (d, d)))

    def rows(s, e):
        t = h * torch.arange(s, e, dtype=F64, device=DEV)[:, None, None]
        return P * torch.special.ndtr((torch.log(t) - mu) / sig)  # log 0 = -inf: Q(0) = 0

    return rows


def _minus_identity(q):
    A = q.neg_()
    A[0] += torch.eye(A.shape[1], dtype=F64, device=DEV)
    return A


def _model(model, g, d, N):
    """A = e0 - q (Weibull, Gamma) or e0 - Qbar_h (Lognormal, endpoint mean-value rule)."""
    if model == "gamma":
        return _minus_identity(_gamma_q(g, N))
    if model == "weibull":
        return _minus_identity(_weibull_q(g, d, N))
    Q = _lognormal_Q(g, d, N)
    A = torch.empty((N, d, d), dtype=F64, device=DEV)
    for s, e in _rows(N, d):  # Qbar(m) = (dQ(m) + dQ(m+1)) / 2, dQ(0) = 0
        x = Q(max(s - 1, 0), e + 1)
        if s == 0:
            x = torch.cat([x[:1], x])
        A[s:e] = (x[2:] - x[:-2]) * 0.5
    return _minus_identity(A)


def _batch_shapes(case, seed):
    """The models' sizes belong to the case (a rerun has the same models in
    hand), their parameters to the seed."""
    g = _rng(case["n"] * 1000 + case["dhi"], 7)
    return [(int(g.integers(case["dlo"], case["dhi"] + 1)), int(round(2.0 ** g.uniform(case["lo"], case["hi"]))))
            for _ in range(case["n"])]


def _inputs(case, seed):
    kind, g = case["kind"], _rng(seed, 1)
    if kind == "inverse":
        return {"A": _model(case["model"], g, case["d"], case["N"])}
    if kind == "batch":
        return {"As": [_model("weibull" if b % 2 == 0 else "lognormal", _rng(seed, 100 + b), d, N)
                       for b, (d, N) in enumerate(_batch_shapes(case, seed))]}
    d, N = case["d"], case["N"]
    if kind == "mre":
        if case["model"] == "exponential":
            G = np.array([[-0.2, 0.2, 0.0, 0.0], [0.01, -0.11, 0.1, 0.0], [0.15, 0.3, -0.85, 0.4],
                          [0.0, 0.0, 0.5, -0.5]]) * g.uniform(0.9, 1.1)
            a = -np.diag(G)
            P = G / a[:, None]
            np.fill_diagonal(P, 0.0)
            t = 0.005 * torch.arange(N + 1, dtype=F64, device=DEV)[:, None]
            Q = _dev(P)[None] * (1.0 - torch.exp(-t * _dev(a)))[:, :, None]
        else:
            Q = _lognormal_Q(g, d, N)(0, N + 1)
        return {"Q": Q, "L": torch.diag_embed(1.0 - Q[:N].sum(dim=2))}
    q = _weibull_q(g, d, N)
    if kind == "entrance":
        D = list(range(d - case["nD"], d))
        alpha = torch.full((d - case["nD"],), 1.0 / (d - case["nD"]), dtype=F64, device=DEV)
        return {"q": q, "D": D, "alpha": alpha}
    alpha = g.uniform(0.0, 1.0, d)
    return {"q": q, "psi": _newton64(_minus_identity(q.clone())), "alpha": _dev(alpha / alpha.sum()),
            "up": list(range(0, max(1, (3 * d) // 4))), "r": _dev(g.uniform(0.0, 1.0, (N, d, case["c"])))}


def prepare(case, seed):
    state = {"case": case, **_inputs(case, seed)}
    if case["kind"] == "batch":
        # a program that runs a batch again and again keeps its result buffers
        state["outs"] = [torch.empty_like(a) for a in state["As"]]
    return state


# ---------------------------------------------------------------------------
# one pass

def run(state):
    case = state["case"]
    kind, prec = case["kind"], case["prec"]
    if kind == "inverse":
        return mrc.inverse(state["A"], prec=prec, sweeps=case.get("sweeps", 1))
    if kind == "batch":
        return mrc.inverse_batched(state["As"], prec=prec, sweeps=case["sweeps"], outs=state["outs"])
    if kind == "mre":
        return mrc.mre_solve(state["Q"], state["L"], scheme="mean_value", prec=prec)
    if kind == "entrance":
        return mrc.first_entrance(state["q"], state["D"], state["alpha"], prec=prec)
    P = mrc.transition(state["psi"], state["q"], prec=prec)
    return {"P": P, "availability": mrc.occupation(P, state["alpha"], state["up"]),
            "visits": mrc.renewal_visits(state["psi"], state["alpha"], state["up"]),
            "V": mrc.reward(state["psi"], state["r"], prec=prec)}


# ---------------------------------------------------------------------------
# what a pass cannot do without

def _inverse_flops(d, N, sweeps=0):
    """Newton doubling by FFT: per level m five real transforms of 2 m points
    per entry and two products of d x d matrices at m + 1 frequencies; a
    refinement sweep takes the same on 2 pow2ceil(N) points."""
    def stage(m):
        return 5 * 2.5 * 2 * m * math.log2(2 * m) * d * d + 2 * 8.0 * d ** 3 * (m + 1)
    f, m = 2.0 * d ** 3, 1
    while m < N:
        f += stage(m)
        m *= 2
    return f + sweeps * stage(m)


def _product_flops(r, m, c, N):
    M = 1 << max(0, (N - 1).bit_length())
    return 2.5 * 2 * M * math.log2(2 * M) * (r * m + m * c + r * c) + 8.0 * r * m * c * (M + 1)


def work(case):
    kind = case["kind"]
    if kind == "batch":
        shapes = _batch_shapes(case, 0)
        sw = case["sweeps"] if case["prec"] == "mixed" else 0
        return {"bytes": sum(16.0 * N * d * d for d, N in shapes),
                "flops": sum(_inverse_flops(d, N, sw) for d, N in shapes)}
    d, N = case["d"], case["N"]
    sw = case.get("sweeps", 1) if case["prec"] == "mixed" else 0
    if kind == "inverse":
        return {"bytes": 16.0 * N * d * d, "flops": _inverse_flops(d, N, sw)}
    if kind == "mre":
        return {"bytes": 24.0 * N * d * d, "flops": _inverse_flops(d, N, sw) + _product_flops(d, d, d, N)}
    if kind == "entrance":
        nD = case["nD"]
        nC = d - nD
        return {"bytes": 8.0 * N * (d * d + nC * nD + 2), "flops": _inverse_flops(nC, N, sw) + _product_flops(nC, nC, nD, N)}
    c = case["c"]
    return {"bytes": 8.0 * N * (3 * d * d + 2 * d * c + 2),
            "flops": _product_flops(d, d, c, N) + 2.5 * 2 * N * math.log2(2 * N) * (2 * d * d + d) + 6.0 * d * d * N}


# ---------------------------------------------------------------------------
# the same results from torch's FP64 transforms and products alone

def _spectrum(x, L):
    return torch.fft.rfft(x, n=L, dim=0)


def _matmul_(X, Y):
    """X(f) Y(f) for square X, written over X in frequency ranges."""
    step = max(1, (1 << 24) // (X.shape[1] * X.shape[2]))
    for s in range(0, X.shape[0], step):
        X[s:s + step] = X[s:s + step] @ Y[s:s + step]
    return X


def _newton64(A):
    """A^(-1) mod x^N: B <- B (2 - A B), the level's products cyclic of length 2 n."""
    N = A.shape[0]
    B = torch.zeros_like(A)
    B[0] = torch.linalg.inv(A[0])
    n = 1
    while n < N:
        m = min(2 * n, N)
        Bh = _spectrum(B[:n], 2 * n)
        E = torch.fft.irfft(_matmul_(_spectrum(A[:m], 2 * n), Bh), n=2 * n, dim=0)[n:].neg()
        Rh = _spectrum(E, 2 * n)
        del E
        for s in range(0, Rh.shape[0], 4096):
            Rh[s:s + 4096] = Bh[s:s + 4096] @ Rh[s:s + 4096]
        del Bh
        B[n:m] = torch.fft.irfft(Rh, n=2 * n, dim=0)[:m - n]
        del Rh
        n *= 2
    return B


def _convolve64(X, Y):
    N = X.shape[0]
    L = 2 << max(0, (N - 1).bit_length())
    return torch.fft.irfft(_spectrum(X, L) @ _spectrum(Y, L), n=L, dim=0)[:N].clone()


def exact(case, seed):
    s, kind = _inputs(case, seed), case["kind"]
    if kind == "inverse":
        return _newton64(s["A"])
    if kind == "batch":
        return [_newton64(a) for a in s["As"]]
    if kind == "mre":
        Q, L = s["Q"], s["L"]
        N, d = L.shape[0], L.shape[1]
        dQ = Q[1:] - Q[:-1]  # dQ[m] = Delta+ Q(m)
        bar = dQ * 0.5
        bar[1:] += dQ[:-1] * 0.5
        return _convolve64(_newton64(_minus_identity(bar)), L - 0.5 * (dQ[:N] @ L[0]))
    if kind == "entrance":
        q, D = s["q"], s["D"]
        C = [i for i in range(q.shape[1]) if i not in D]
        gm = _convolve64(_newton64(_minus_identity(q[:, C][:, :, C].clone())), q[:, C][:, :, D])
        F = torch.cumsum((s["alpha"][None, :, None] * gm).sum(dim=(1, 2)), dim=0)
        return gm, F, 1.0 - F
    psi, q, up = s["psi"], s["q"], s["up"]
    N = q.shape[0]
    L = 2 << max(0, (N - 1).bit_length())
    H = 1.0 - torch.cumsum(q.sum(dim=2), dim=0)
    P = torch.fft.irfft(_spectrum(psi, L) * _spectrum(H, L)[:, None, :], n=L, dim=0)[:N].clone()
    occ = (P[:, :, up].sum(dim=2) * s["alpha"]).sum(dim=1)
    vis = torch.cumsum((psi[:, :, up].sum(dim=2) * s["alpha"]).sum(dim=1), dim=0)
    return {"P": P, "availability": occ, "visits": vis, "V": _convolve64(psi, s["r"])}
