"""Workspace of the supernodal route: what a solve keeps beside x itself (update vectors,
backward partials) is bounded however many value sets and right-hand sides there are."""
import pytest

from paper_2609_29765_gb300 import inputs as I
from paper_2609_29765_gb300.api import Plan


@pytest.mark.parametrize("dims", [(12, 12, 12, 5), (20, 20, 20, 20)])
def test_workspace_per_chain(dims):
    Ap, Ai, coords = I.stcov_pattern(*dims)
    n = len(Ap) - 1
    P = Plan(n, Ap, Ai, coords=coords, nb=64, route="supernodal")
    # from some number of chains on, a chain more is one vector of n and its step flags: four
    # ints a supernode or chunk at most, and there are no more of those than 3 n / 4
    assert P.workspace_bytes(40000) - P.workspace_bytes(20000) <= 20000 * (8 * n + 12 * n)
    # 256 MB at most, or 32 chains
    one = P.workspace_bytes(1)
    assert P.workspace_bytes(40000) <= 40000 * 20 * n + max(32 * one, 256 << 20) + 4096
