"""GPU tests of the supernodal solve on the elimination tree: panels with more rows below
than one chunk holds, many children, several roots, several right-hand sides and value
sets, against the oracle."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2609_29765_gb300 import inputs as I

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _blocks(seed):
    import scipy.sparse as sp
    parts = []
    for k, n in enumerate((1, 40, 300, 7)):
        Ap, Ai, Ax = I.random_spd(n, 0.5, seed=seed + k)
        L = sp.csc_matrix((Ax, Ai, Ap), shape=(n, n))
        parts.append(L + sp.tril(L, -1).T)
    return I.lower_csc(sp.block_diag(parts, format="csc"))


# rows below a panel: 256-row chunks, so 128 + 256, one more, and several chunks
CASES = {
    "dense 384": lambda: I.random_spd(384, 0.9, seed=1),
    "dense 385": lambda: I.random_spd(385, 0.9, seed=2),
    "dense 900": lambda: I.random_spd(900, 0.7, seed=3),
    "band 1200, half-bandwidth 310": lambda: I.band(1200, 310, seed=4),
    "arrowhead, 3000 children": lambda: I.arrowhead(3000, 20, seed=5),
    "disconnected blocks": lambda: _blocks(6),
}


@pytest.mark.parametrize("name", list(CASES))
@pytest.mark.parametrize("batch,nrhs", [(1, 1), (3, 2)])
def test_solve(name, batch, nrhs):
    from paper_2609_29765_gb300.api import Plan
    Ap, Ai, Ax = CASES[name]()
    n = len(Ap) - 1
    P = Plan(n, Ap, Ai, nb=64, route="supernodal", ordering="natural")
    scale = 1.0 + np.arange(batch)
    fac = P.factorize(torch.as_tensor(scale[:, None] * Ax, device="cuda"), check_status=True)
    b = I.rhs(n, 7, batch * nrhs).reshape(batch, nrhs, n)
    x = fac.solve(torch.as_tensor(b, device="cuda")).cpu().numpy()
    assert fac.status() == 0
    F = O.OracleFactor(n, Ap, Ai, P.export("perm"))
    for k in range(batch):
        Lo, info = F.factor(scale[k] * Ax)
        assert info == 0
        for r in range(nrhs):
            xo = F.solve(Lo, b[k, r])
            assert np.linalg.norm(x[k, r] - xo) <= 1e-10 * np.linalg.norm(xo)
