"""The list filter at the shapes with many representatives, against an optimum that
is known: K clusters far apart, each of few distinct points that repeat.  A set of
centers without a center in some cluster costs at least the separation, so the
optimum has one in each, and its value is the largest over the clusters of the
smallest radius of a member.  A filter that dropped a sample that matters would
certify a smaller optimum or a bound above this one."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2301_00061_gb300 import KCenter  # noqa: E402


def _instance(n, d, k, m, seed):
    rng = np.random.default_rng(seed)
    corners = 60.0 * np.array([[(i >> a) & 1 for a in range(d)] for i in range(2 ** d)])
    at = corners[rng.choice(2 ** d, k, replace=False)] if 2 ** d >= k else 60.0 * np.arange(k)[:, None] + np.zeros(d)
    pts = (at[:, None] + rng.uniform(-2, 2, (k, m, d))).astype(np.float32)
    P = pts.astype(np.float64)
    r2 = ((P[:, :, None] - P[:, None]) ** 2).sum(-1).max(-1)   # radius of each member as a center
    optimum = float(r2.min(1).max())
    assert optimum < 30.0 ** 2
    flat = pts.reshape(-1, d)
    X = flat[np.concatenate([np.arange(k * m), rng.integers(0, k * m, n - k * m)])]
    return X[rng.permutation(n)], optimum


# lists are filtered from 2048 entries on; work items of 1024
# (drops: the filter shortens lists on the way; the one instance closes before that)
@pytest.mark.parametrize("n,d,k,m,drops", [(2_049, 8, 8, 30, True), (5_000, 8, 5, 60, True), (3_073, 7, 6, 40, False),
                                           (3_073, 7, 6, 90, True), (9_001, 5, 7, 50, True), (4_097, 6, 3, 200, True),
                                           (20_000, 4, 4, 400, True), (6_000, 3, 4, 300, True),
                                           (10_000, 2, 3, 900, True)])
def test_known_optimum(n, d, k, m, drops):
    X, optimum = _instance(n, d, k, m, n + d)
    with KCenter(torch.from_numpy(X).cuda(), k) as kc:
        for limit in (0, 4, 64):   # to the certificate, and the bounds on the way
            r = kc.solve(tol=1e-12, lists=1, node_limit=limit, time_limit_s=60.0)
            assert r["lower_bound"] <= optimum * (1 + 1e-12)
            assert r["objective"] >= optimum * (1 - 1e-12)
            assert oracle.objective(X, r["centers"])[0] == r["objective"]
            if limit == 0:
                assert r["status"] == 0 and abs(r["objective"] - optimum) <= 1e-12 * optimum
                assert (r["lists_filtered"] > 0 and r["samples_dropped"] > 0) or not drops
