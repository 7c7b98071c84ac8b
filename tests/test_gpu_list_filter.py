"""The list filter's staging at the sizes where it can go wrong: lists of one
entry up to several work items of 1,024, with every compiled attribute count and
with the representatives of K = 8 at D = 8 (its static and dynamic shared memory
together exceed 48 KiB)."""
import numpy as np
import pytest

import oracle
from paper_2301_00061_gb300 import KCenter

pytestmark = pytest.mark.gpu


def _blobs(n, d, k, seed):
    rng = np.random.default_rng(seed)
    means = rng.uniform(0.0, 20.0, (k, d))
    return (means[rng.integers(0, k, n)] + rng.normal(size=(n, d))).astype(np.float32)


@pytest.mark.parametrize("n,d,k", [(33, 2, 2), (1025, 2, 3), (2049, 4, 3), (1023, 3, 4), (3000, 6, 2)])
def test_lists_equal_shared_set(n, d, k):
    """Dropping redundant samples loses nothing: with and without lists a solve
    certifies the same optimum (both are the objective of a center set in double,
    so they are equal), and it is the oracle's."""
    import torch
    X = _blobs(n, d, k, seed=n)
    with KCenter(torch.from_numpy(X).cuda(), k) as kc:
        a = kc.solve(tol=1e-12, lists=1)
        b = kc.solve(tol=1e-12, lists=0)
    assert a["status"] == b["status"] == 0
    assert abs(a["objective"] - b["objective"]) <= 1e-12 * b["objective"]
    assert oracle.objective(X, a["centers"])[0] == a["objective"]


@pytest.mark.parametrize("d,k", [(8, 8), (7, 6), (8, 5)])
def test_lists_with_many_representatives(d, k):
    """A bounded number of nodes: the objective is that of its centers, and the
    lower bound does not pass it."""
    import torch
    X = _blobs(3000, d, k, seed=d * k)
    with KCenter(torch.from_numpy(X).cuda(), k) as kc:
        g = kc.solve(tol=1e-12, lists=1, node_limit=256)
    assert g["lower_bound"] <= g["objective"]
    assert oracle.objective(X, g["centers"])[0] == g["objective"]
