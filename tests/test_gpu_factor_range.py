"""GPU tests of the factorization where rows and pivots differ in scale: graded rows that the
split products take as they are, and positive pivots on both sides of the range of the 16-column
diagonal blocks' fast path ([2^-991, 2^989)), against the oracle."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2609_29765_gb300 import inputs as I

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
ROUTES = ["supernodal", "semisparse", "dense"]


def _check(Ap, Ai, Ax, u, nb, route, **kw):
    """L of D A D, D = diag(2^u) (exact), row i over 2^u_i, against the oracle's L of A: 1e-11
    of a column's largest entry, the factor tolerance of every route."""
    from paper_2609_29765_gb300.api import Plan
    n = len(Ap) - 1
    col = np.repeat(np.arange(n), np.diff(Ap))
    P = Plan(n, Ap, Ai, nb=nb, route=route, **kw)
    fac = P.factorize(torch.as_tensor(np.ldexp(Ax, u[Ai] + u[col])[None], device="cuda"), check_status=True)
    assert int(fac.info[0]) == 0
    Lp, Li = P.export("Lp"), P.export("Li")
    perm = P.export("perm")
    L = np.ldexp(fac.to_csc().cpu().numpy()[0], -u[perm][Li])
    F = O.OracleFactor(n, Ap, Ai, perm)
    Lo, info = F.factor(Ax)
    assert info == 0
    cm = np.maximum.reduceat(np.abs(Lo), Lp[:-1])
    assert np.all(np.abs(L - Lo) <= 1e-11 * np.repeat(cm, np.diff(Lp)))
    ld = F.logdet(Lo) + 2.0 * np.log(2.0) * float(u.sum())
    assert abs(float(fac.logdet()[0]) - ld) <= 1e-10 * max(1.0, abs(ld))


def _stcov():
    Ap, Ai, coords = I.stcov_pattern(9, 8, 7, 3)
    return Ap, Ai, I.stcov_values((1.3, 0.6, 0.4), 9, 8, 7, 3), dict(coords=coords, nb=64)


MATRICES = {
    "stcov": _stcov,
    "dense 200": lambda: (*I.random_spd(200, 0.9, seed=3), dict(ordering="natural", nb=128)),
    "band": lambda: (*I.band(300, 70, seed=4), dict(ordering="natural", nb=64)),
}


# every row of L inside 2^+-400: all chunks are split products
@pytest.mark.parametrize("route", ROUTES)
@pytest.mark.parametrize("name", list(MATRICES))
def test_graded_rows_in_range(name, route):
    Ap, Ai, Ax, kw = MATRICES[name]()
    u = np.random.default_rng(1).integers(-300, 301, size=len(Ap) - 1)
    _check(Ap, Ai, Ax, u, kw.pop("nb"), route, **kw)


# pivots near 2^989 and 2^-991 (of A: 2^(2 u)), some on either side in one block
@pytest.mark.parametrize("route", ROUTES)
@pytest.mark.parametrize("lo,hi", [(490, 499), (498, 503), (-499, -490), (-505, -499)])
@pytest.mark.parametrize("name", list(MATRICES))
def test_pivots_out_of_range(name, lo, hi, route):
    Ap, Ai, Ax, kw = MATRICES[name]()
    u = np.random.default_rng(2).integers(lo, hi + 1, size=len(Ap) - 1)
    _check(Ap, Ai, Ax, u, kw.pop("nb"), route, **kw)
