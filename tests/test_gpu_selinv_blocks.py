"""GPU tests of the selected inverse's diagonal blocks at the edges of their 16-column panels
and of the width up to which the panels' inverses fit beside the block (112), against the
dense inverse."""
import numpy as np
import pytest

from paper_2609_29765_gb300 import inputs as I

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("route", ["supernodal", "semisparse", "dense"])
@pytest.mark.parametrize("n", [1, 15, 17, 32, 33, 111, 112, 113, 128, 200])
def test_dense_block(route, n):
    from paper_2609_29765_gb300.api import Plan
    Ap, Ai, Ax = I.random_spd(n, 0.9 if n > 1 else 0.0, seed=n)
    P = Plan(n, Ap, Ai, nb=128, route=route, ordering="natural")
    fac = P.factorize(torch.as_tensor(np.stack([Ax, 3.0 * Ax]), device="cuda"), check_status=True)
    g = fac.logdet_backward().cpu().numpy()
    col = np.repeat(np.arange(n), np.diff(Ap))
    A = np.zeros((n, n))
    A[Ai, col] = Ax
    A[col, Ai] = Ax
    S = np.linalg.inv(A)
    want = S[Ai, col] * np.where(Ai == col, 1.0, 2.0)
    for b, s in enumerate((1.0, 3.0)):
        assert np.max(np.abs(g[b] - want / s)) <= 1e-11 * np.max(np.abs(S)) / s


# a band inside one block: entries outside the band stay out of the recurrence
@pytest.mark.parametrize("bw", [1, 5, 15, 16, 40])
def test_band_in_a_block(bw):
    from paper_2609_29765_gb300.api import Plan
    n = 90
    Ap, Ai, Ax = I.band(n, bw, seed=bw)
    P = Plan(n, Ap, Ai, nb=64, route="semisparse", ordering="natural")
    fac = P.factorize(torch.as_tensor(Ax, device="cuda")[None], check_status=True)
    g = fac.logdet_backward().cpu().numpy()[0]
    col = np.repeat(np.arange(n), np.diff(Ap))
    A = np.zeros((n, n))
    A[Ai, col] = Ax
    A[col, Ai] = Ax
    S = np.linalg.inv(A)
    assert np.max(np.abs(g - S[Ai, col] * np.where(Ai == col, 1.0, 2.0))) <= 1e-11 * np.max(np.abs(S))
