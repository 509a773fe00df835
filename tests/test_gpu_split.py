"""GPU tests of the split (exact integer) tile products: matrices whose scale leaves the
range the split accepts (those chunks are multiplied with DFMAs), rows and pivots of very
different magnitude, and ragged cells, element by element against the oracle."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2609_29765_gb300 import inputs as I

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _check(n, Ap, Ai, Ax, coords, nb, route, d=None, **kw):
    """Factors of D A D and 2 D A D, D = diag(d), d powers of two: scaling by powers of two is
    exact, so L(D A D) = D L(A), and row i of the result over d_i is compared."""
    from paper_2609_29765_gb300.api import Plan
    P = Plan(n, Ap, Ai, coords=coords, nb=nb, route=route, **kw)
    d = np.ones(n) if d is None else d
    vals = Ax * d[Ai] * d[np.repeat(np.arange(n), np.diff(Ap))]
    vals = torch.as_tensor(np.stack([vals, 2.0 * vals]), device="cuda")
    fac = P.factorize(vals, check_status=True)
    assert int(fac.info.abs().sum()) == 0
    Lg = fac.to_csc().cpu().numpy()
    Lp, Li = P.export("Lp"), P.export("Li")
    dp = d[P.export("perm")]
    F = O.OracleFactor(n, Ap, Ai, P.export("perm"))
    for b, s in enumerate((1.0, 2.0)):
        Lo, info = F.factor(s * Ax)
        assert info == 0
        cm = np.maximum.reduceat(np.abs(Lo), Lp[:-1])
        # 1e-11 of the column's largest entry: the factor tolerance of every route
        assert np.all(np.abs(Lg[b] / dp[Li] - Lo) <= 1e-11 * np.repeat(cm, np.diff(Lp)))
        ld = F.logdet(Lo) + 2.0 * float(np.log(d).sum())
        assert abs(float(fac.logdet()[b]) - ld) <= 1e-10 * max(1.0, abs(ld))


# 2^400 bounds the rows of L the split takes: A scaled by 2^-840 and 2^840 leaves it (DFMA
# chunks), 2^-700 and 2^700 does not
@pytest.mark.parametrize("route", ["supernodal", "semisparse", "dense"])
@pytest.mark.parametrize("scale", [-420, -350, 350, 420])
def test_uniform_scale(route, scale):
    Ap, Ai, Ax, coords = I.laplace2d_bordered(19, 23, 3)
    n = len(Ap) - 1
    _check(n, Ap, Ai, Ax, coords, 64, route, d=np.full(n, 2.0 ** scale))


@pytest.mark.parametrize("route", ["supernodal", "semisparse", "dense"])
def test_graded_rows(route):
    # D A D with D = 2^u, u in [-450, 450]: rows inside and outside the range side by side
    Ap, Ai, coords = I.stcov_pattern(9, 8, 7, 3)
    Ax = I.stcov_values((1.3, 0.6, 0.4), 9, 8, 7, 3)
    n = len(Ap) - 1
    u = np.random.default_rng(3).integers(-450, 451, size=n)
    _check(n, Ap, Ai, Ax, coords, 64, route, d=np.exp2(u.astype(float)))


@pytest.mark.parametrize("route", ["supernodal", "semisparse", "dense"])
def test_graded_pivots(route):
    # diagonals spread over 1e0..1e12: entries of one row of L differ by many orders
    Ap, Ai, Ax, coords = I.fem3d(9, 8, 7, seed=4)
    n = len(Ap) - 1
    Ax = Ax.copy()
    Ax[Ap[:-1]] += 10.0 ** np.random.default_rng(5).uniform(0, 12, size=n)
    _check(n, Ap, Ai, Ax, coords, 64, route)


# cells and tiles of every remainder of the 16 x 8 product units and 16-column chunks
@pytest.mark.parametrize("n", [17, 65, 127, 130, 143, 200, 261])
@pytest.mark.parametrize("route", ["supernodal", "semisparse", "dense"])
def test_ragged_dense(route, n):
    Ap, Ai, Ax = I.random_spd(n, 0.6, seed=n)
    _check(n, Ap, Ai, Ax, None, 128, route, ordering="natural")


# tau = 2 makes sums of products that end just below a power of two (53 leading ones): the
# rounding of an exact sum has to carry into the exponent
@pytest.mark.parametrize("route", ["supernodal", "semisparse", "dense"])
@pytest.mark.parametrize("theta", [(2.0, 0.6, 0.7), (0.5, 0.5, 1.0), (8.0, 0.25, 1.0)])
def test_sums_below_powers_of_two(route, theta):
    dims = (14, 12, 8, 0)
    Ap, Ai, coords = I.stcov_pattern(*dims)
    _check(len(Ap) - 1, Ap, Ai, I.stcov_values(theta, *dims), coords, 32, route)
