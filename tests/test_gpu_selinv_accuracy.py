"""GPU tests of the selected inverse's accuracy: Sigma and the logdet gradient for the factor
that the GPU returns, against L^{-T} L^{-1} in extended precision, over sqrt(Sigma_ii Sigma_jj)
(so independent of the units of the variables).

Tolerance: the element recurrence (one column at a time, plain FP64) restated here is run on
the same factor, and the kernels may have 8 times its error -- the same recurrence summed in
another order -- plus 64 eps for the roundings that do not grow with the conditioning.
"""
import numpy as np
import pytest

from paper_2609_29765_gb300 import inputs as I

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
ROUTES = ["supernodal", "semisparse", "dense"]


def _extended(L):
    n = len(L)
    L = L.astype(np.longdouble)
    W = np.zeros((n, n), dtype=np.longdouble)
    for i in range(n):
        W[i, i] = 1
        W[i] -= L[i, :i] @ W[:i]
        W[i] /= L[i, i]
    return W.T @ W


def _recurrence(L):
    n = len(L)
    S = np.zeros((n, n))
    for c in range(n - 1, -1, -1):
        l, inv = L[c + 1:, c], 1.0 / L[c, c]
        S[c + 1:, c] = -(S[c + 1:, c + 1:] @ l) * inv
        S[c, c + 1:] = S[c + 1:, c]
        S[c, c] = inv * inv - (l @ S[c + 1:, c]) * inv
    return S


def _check(Ap, Ai, Ax, nb, route, d=None, **kw):
    """D A D with D = diag(d) of powers of two (exact); row i of L over d_i and d_i Sigma_ij d_j
    are those of A's own scale."""
    from paper_2609_29765_gb300.api import Plan
    n = len(Ap) - 1
    col = np.repeat(np.arange(n), np.diff(Ap))
    d = np.ones(n) if d is None else d
    P = Plan(n, Ap, Ai, nb=nb, route=route, **kw)
    fac = P.factorize(torch.as_tensor((Ax * d[Ai] * d[col])[None], device="cuda"), check_status=True)
    assert int(fac.info[0]) == 0
    perm = P.export("perm")
    ip = np.empty(n, dtype=np.int64)
    ip[perm] = np.arange(n)
    Lp, Li = P.export("Lp"), P.export("Li")
    Lc, dp = np.repeat(np.arange(n), np.diff(Lp)), d[perm]
    L = np.zeros((n, n))
    L[Li, Lc] = fac.to_csc().cpu().numpy()[0] / dp[Li]
    S = _extended(L)
    sd = np.sqrt(np.diag(S).astype(np.float64))

    def err(rows, cols, got):
        return float(np.max(np.abs(got - S[rows, cols]) / (sd[rows] * sd[cols])))

    tol = 8.0 * err(Li, Lc, _recurrence(L)[Li, Lc]) + 64 * np.finfo(float).eps
    assert err(Li, Lc, fac.selinv().to_csc().cpu().numpy()[0] * dp[Li] * dp[Lc]) <= tol
    g = fac.logdet_backward().cpu().numpy()[0] * d[Ai] * d[col] / np.where(Ai == col, 1.0, 2.0)
    assert err(ip[Ai], ip[col], g) <= tol


def _grid():
    Ap, Ai, Ax, coords = I.laplace2d_bordered(15, 16, 3)
    return Ap, Ai, Ax, dict(coords=coords, nb=64)


def _stcov():
    Ap, Ai, coords = I.stcov_pattern(7, 6, 6, 3)
    return Ap, Ai, I.stcov_values((1.3, 0.6, 0.4), 7, 6, 6, 3), dict(coords=coords, nb=32)


MATRICES = {
    "dense 150": lambda: (*I.random_spd(150, 0.9, seed=2), dict(nb=128, ordering="natural")),
    "dense 200": lambda: (*I.random_spd(200, 0.9, seed=3), dict(nb=64, ordering="natural")),
    "band": lambda: (*I.band(260, 40, seed=4), dict(nb=64, ordering="natural")),
    "narrow band": lambda: (*I.band(200, 20, seed=5), dict(nb=32, ordering="natural")),
    "grid": _grid,
    "stcov": _stcov,
}


# one variable in other units, then all of them; 2^+-350 is beyond the balance the split takes
# (those chunks are DFMAs)
@pytest.mark.parametrize("route", ROUTES)
@pytest.mark.parametrize("units", ["one 2^20", "one 2^40", "all 2^30", "all 2^100", "all 2^350"])
@pytest.mark.parametrize("name", list(MATRICES))
def test_units(name, units, route):
    Ap, Ai, Ax, kw = MATRICES[name]()
    n = len(Ap) - 1
    which, e = units.split(" 2^")
    u = np.zeros(n)
    if which == "one":
        u[n // 2] = float(e)
    else:
        u = np.random.default_rng(n).integers(-int(e), int(e) + 1, size=n).astype(float)
    _check(Ap, Ai, Ax, kw.pop("nb"), route, d=np.exp2(u), **kw)


# ---- intrinsic fields and covariance kernels with a small ridge: ill-conditioned panels ----
def _dense_lower(A, bw=None):
    import scipy.sparse as sp
    A = np.where(np.abs(np.subtract.outer(np.arange(len(A)), np.arange(len(A)))) <= (len(A) if bw is None else bw), A, 0.0)
    return I.lower_csc(sp.csc_matrix(A))


def _walk(n, order, ridge):
    D = np.eye(n)
    for _ in range(order):
        D = np.diff(D, axis=0)
    return D.T @ D + ridge * np.eye(n)


def _kernel(n, f, ridge):
    r = np.abs(np.subtract.outer(np.arange(n), np.arange(n))).astype(float)
    return f(r) + ridge * np.eye(n)


def _matern(r, length=20.0):
    s = np.sqrt(5.0) * r / length
    return (1.0 + s + s * s / 3.0) * np.exp(-s)


RIDGED = {
    "walk of order 1 + 1e-8": lambda: (_walk(96, 1, 1e-8), 1),
    "walk of order 2 + 1e-8": lambda: (_walk(96, 2, 1e-8), 2),
    "walk of order 3 + 1e-8": lambda: (_walk(96, 3, 1e-8), 3),
    "Matern 5/2, range 20, + 1e-8": lambda: (_kernel(96, _matern, 1e-8), None),
    "squared exponential, range 3, + 1e-8": lambda: (_kernel(96, lambda r: np.exp(-r * r / 18.0), 1e-8), None),
    "squared exponential, range 3, + 1e-10": lambda: (_kernel(96, lambda r: np.exp(-r * r / 18.0), 1e-10), None),
}


# blocks up to 112 columns with and without the panels' inverses; in other units, too
@pytest.mark.parametrize("route", ROUTES)
@pytest.mark.parametrize("nb", [32, 64, 128])
@pytest.mark.parametrize("units", [0, 30])
@pytest.mark.parametrize("name", list(RIDGED))
def test_ridged(name, units, nb, route):
    A, bw = RIDGED[name]()
    Ap, Ai, Ax = _dense_lower(A, bw)
    u = np.random.default_rng(nb).integers(-units, units + 1, size=len(A)).astype(float)
    _check(Ap, Ai, Ax, nb, route, d=np.exp2(u), ordering="natural")
