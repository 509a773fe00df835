"""GPU tests of the two supernodal solves: chains of supernodes (gathered row by row), wide
trees with panels of several chunks (update vectors), and the same patterns with few and with
many right-hand sides, against the oracle."""
import numpy as np
import pytest
import scipy.sparse as sp

from oracle import oracle as O
from paper_2609_29765_gb300 import inputs as I

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _bordered(blocks, size, border):
    """Dense blocks tied by dense border rows: chains of panels with up to size + border rows
    below, and a root with cells of every panel."""
    rng = np.random.default_rng(size)
    A = sp.block_diag([sp.csc_matrix(rng.uniform(-1, 1, (size, size)) / size) for _ in range(blocks)], format="csc")
    B = sp.csc_matrix(rng.uniform(-1, 1, (border, blocks * size)) / size)
    M = sp.bmat([[A + A.T, B.T], [B, sp.csc_matrix((border, border))]], format="csc")
    M = M + sp.diags(1.0 + np.asarray(abs(M).sum(axis=0)).ravel())
    return (*I.lower_csc(M), dict(ordering="natural"))


CASES = {
    "dense 130": lambda: (*I.random_spd(130, 0.9, seed=1), dict(ordering="natural")),
    "dense 700": lambda: (*I.random_spd(700, 0.9, seed=2), dict(ordering="natural")),
    "band 900, half-bandwidth 200": lambda: (*I.band(900, 200, seed=3), dict(ordering="natural")),
    "band 1500, half-bandwidth 8": lambda: (*I.band(1500, 8, seed=4), dict(ordering="natural")),
    "random, RCM": lambda: (*I.random_spd(600, 0.008, seed=5), dict(ordering="rcm")),
    "16 blocks of 420, border 60": lambda: _bordered(16, 420, 60),
    "3 blocks of 5, border 1": lambda: _bordered(3, 5, 1),
}


@pytest.mark.parametrize("name", list(CASES))
@pytest.mark.parametrize("batch,nrhs", [(1, 1), (2, 3), (1, 700)])
def test_solve(name, batch, nrhs):
    from paper_2609_29765_gb300.api import Plan
    Ap, Ai, Ax, kw = CASES[name]()
    n = len(Ap) - 1
    P = Plan(n, Ap, Ai, nb=64, route="supernodal", **kw)
    scale = 1.0 + np.arange(batch)
    fac = P.factorize(torch.as_tensor(scale[:, None] * Ax, device="cuda"), check_status=True)
    b = I.rhs(n, 7, batch * nrhs).reshape(batch, nrhs, n)
    x = fac.solve(torch.as_tensor(b, device="cuda")).cpu().numpy()
    assert fac.status() == 0
    F = O.OracleFactor(n, Ap, Ai, P.export("perm"))
    for k in range(batch):
        Lo, info = F.factor(scale[k] * Ax)
        assert info == 0
        for r in sorted({0, 1 % nrhs, nrhs // 2, nrhs - 1}):
            xo = F.solve(Lo, b[k, r])
            assert np.linalg.norm(x[k, r] - xo) <= 1e-10 * np.linalg.norm(xo)
