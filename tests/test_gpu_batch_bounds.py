"""Float node bounds of batches (the pruning kernel) and of few nodes (the
streaming kernel) against the FP64 oracle on grid data, where every float
operation is exact: coordinates and boxes are small multiples of 1/4, so the
values are equal bit for bit and the arg-max is the smallest index.

Sizes sit at the edges of the kernels' tiles (128 to 2048 samples), strips,
groups of 8 and 64 nodes, attribute pairs and the switch between the two paths.
"""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2301_00061_gb300 import KCenter  # noqa: E402

DEV = torch.device("cuda:0")


def _t(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to(DEV)


def _grid(n, d, k, b, seed, spread=40):
    """Blobs on a 1/4 grid and boxes of mixed sizes around them, in a shuffled
    cluster order per node (so no cluster is the nearest one everywhere)."""
    rng = np.random.default_rng(seed)
    means = rng.integers(-spread, spread, size=(k, d))
    X = (means[rng.integers(0, k, n)] + np.rint(4 * rng.standard_normal((n, d)))) / 4
    at = np.stack([means[rng.permutation(k)] for _ in range(b)]) / 4
    lo = at - np.rint(rng.integers(0, 24, size=(b, k, d)) * rng.random((b, 1, 1))) / 4
    hi = at + np.rint(rng.integers(0, 24, size=(b, k, d)) * rng.random((b, 1, 1))) / 4
    return X.astype(np.float32), lo.astype(np.float32), hi.astype(np.float32)


def _check(X, k, lo, hi):
    kc = KCenter(_t(X), k)
    lb, raw, arg = (v.cpu().numpy() for v in kc.lower_bounds(_t(lo), _t(hi)))
    ref, refarg = oracle.lower_bounds(X, lo, hi)
    np.testing.assert_array_equal(raw, ref)
    np.testing.assert_array_equal(arg, refarg)
    assert np.all(lb <= ref)
    kc.close()


# one D per attribute-pair count of the kernels, odd and even
@pytest.mark.parametrize("d", [1, 2, 3, 4, 6, 7, 8, 11, 16, 23, 29, 47, 68, 90, 128])
@pytest.mark.parametrize("n,k,b", [(37, 2, 3), (2_049, 5, 70)])
def test_every_width(d, n, k, b):
    _check(*(lambda X, lo, hi: (X, k, lo, hi))(*_grid(n, d, k, b, 100 + d, spread=8)))


@pytest.mark.parametrize("n", [16, 127, 128, 129, 1_023, 1_025, 2_047, 2_048, 4_097, 700_001])
@pytest.mark.parametrize("b", [1, 2, 4, 9, 65])
def test_tile_edges(n, b):
    _check(*(lambda X, lo, hi: (X, 3, lo, hi))(*_grid(n, 4, 3, b, n + b)))


@pytest.mark.parametrize("k", [1, 2, 3, 4, 5, 9, 16])
@pytest.mark.parametrize("d", [2, 8])
@pytest.mark.parametrize("b", [1, 3, 8, 64, 300])
def test_clusters_and_nodes(k, d, b):
    _check(*(lambda X, lo, hi: (X, k, lo, hi))(*_grid(5_003, d, k, b, 7 * k + b)))


def test_ties_and_zero_bounds():
    """All samples equal, nodes holding every sample (bound 0) and many samples
    attaining the maximum: the smallest index each time."""
    X, lo, hi = _grid(9_001, 3, 3, 40, 5)
    _check(np.ones_like(X), 3, lo, hi)
    lo[::3], hi[::3] = -100, 100
    _check(X, 3, lo, hi)
    _check(np.tile(X[:37], (60, 1)), 3, lo, hi)
    _check(np.sign(X), 3, lo, hi)


def test_unbounded_and_inverted_boxes():
    """Infinite faces hold every coordinate; an inverted box (lo > hi, an empty
    node) keeps the value max(lo - x, x - hi, 0) per attribute in batches as it
    has it alone."""
    X, lo, hi = _grid(6_007, 4, 3, 48, 11)
    lo[5:9, 1], hi[7:12, 2] = -np.inf, np.inf
    _check(X, 3, lo, hi)
    lo[20:24], hi[20:24] = 1, 0
    kc = KCenter(_t(X), 3)
    batch = [v.cpu().numpy() for v in kc.lower_bounds(_t(lo), _t(hi))]
    for b in range(48):
        one = [v.cpu().numpy()[0] for v in kc.lower_bounds(_t(lo[b:b + 1]), _t(hi[b:b + 1]))]
        assert [v[b] for v in batch] == one, b
    kc.close()


@pytest.mark.parametrize("d,k", [(2, 4), (5, 3), (8, 5), (12, 3), (29, 3)])
def test_batches_equal_single_nodes(d, k):
    """Rounded data: a node's value and sample do not depend on its batch."""
    rng = np.random.default_rng(d)
    n, b = 30_011, 130
    X = (rng.standard_normal((n, d)) + 6 * rng.integers(0, 3, (n, 1))).astype(np.float32)
    c = X[rng.integers(0, n, (b, k))]
    h = np.exp(rng.uniform(np.log(1e-3), np.log(4), (b, k, d))).astype(np.float32)
    kc = KCenter(_t(X), k)
    batch = [v.cpu().numpy() for v in kc.lower_bounds(_t(c - h), _t(c + h))]
    for i in range(0, b, 7):
        one = [v.cpu().numpy()[0] for v in kc.lower_bounds(_t((c - h)[i:i + 1]), _t((c + h)[i:i + 1]))]
        assert [v[i] for v in batch] == one, i
    kc.close()
