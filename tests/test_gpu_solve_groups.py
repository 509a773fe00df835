"""GPU test of the supernodal solve with more (value set, right-hand side) chains than are in
flight together: groups of chains share the places of their update vectors and backward
partials."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2609_29765_gb300 import inputs as I

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _stcov():
    Ap, Ai, coords = I.stcov_pattern(12, 12, 12, 5)
    return Ap, Ai, I.stcov_values((1.3, 0.6, 0.4), 12, 12, 12, 5), dict(coords=coords)


def _blocks():  # dense blocks tied by border rows: panels of two chunks, so backward partials
    import scipy.sparse as sp
    rng = np.random.default_rng(4)
    blocks, size, border = 16, 420, 60
    A = sp.block_diag([sp.csc_matrix(rng.uniform(-1, 1, (size, size)) / size) for _ in range(blocks)], format="csc")
    B = sp.csc_matrix(rng.uniform(-1, 1, (border, blocks * size)) / size)
    M = sp.bmat([[A + A.T, B.T], [B, sp.csc_matrix((border, border))]], format="csc")
    return (*I.lower_csc(M + sp.diags(1.0 + np.asarray(abs(M).sum(axis=0)).ravel())), dict(ordering="natural"))


# chains far beyond one group, the last group not full, by value sets and by right-hand sides
@pytest.mark.parametrize("make,batch,nrhs", [(_stcov, 1, 10001), (_stcov, 3, 3333), (_blocks, 1, 3001), (_blocks, 3, 999)])
def test_groups(make, batch, nrhs):
    from paper_2609_29765_gb300.api import Plan
    Ap, Ai, Ax, kw = make()
    n = len(Ap) - 1
    P = Plan(n, Ap, Ai, nb=64, route="supernodal", **kw)
    ws = P.workspace_bytes
    assert (ws(batch * nrhs) - ws(batch * nrhs // 2)) < 0.8 * (ws(1000) - ws(500)) / 500 * (batch * nrhs / 2)
    scale = 1.0 + np.arange(batch)
    fac = P.factorize(torch.as_tensor(scale[:, None] * Ax, device="cuda"), check_status=True)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(7)
    b = torch.randn(batch, nrhs, n, generator=gen, device="cuda", dtype=torch.float64)
    x = fac.solve(b)
    assert fac.status() == 0
    # every chain's steps are added in one order: the same bits as a few at a time
    for r0 in range(0, nrhs, 500):
        part = fac.solve(b[:, r0:r0 + 500].contiguous())
        assert torch.equal(part, x[:, r0:r0 + 500])
    F = O.OracleFactor(n, Ap, Ai, P.export("perm"))
    for k in range(batch):
        Lo, info = F.factor(scale[k] * Ax)
        assert info == 0
        for r in (0, nrhs // 2, nrhs - 1):
            xo = F.solve(Lo, b[k, r].cpu().numpy())
            assert np.linalg.norm(x[k, r].cpu().numpy() - xo) <= 1e-10 * np.linalg.norm(xo)
