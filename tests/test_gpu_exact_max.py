"""Exact maxima (double bounds, objectives of float and double data) against the
FP64 oracle, bit for bit: the float screen may only dismiss samples that cannot
attain the double maximum.  Sizes cross the direct / screened switch and the
edges of tiles, groups and the streaming screen; data with a large offset, a
large range, exact ties and maxima closer than float precision try the margin."""
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


def _data(n, d, k, seed, dtype):
    rng = np.random.default_rng(seed)
    means = rng.uniform(0, 20, (k, d))
    return (means[rng.integers(0, k, n)] + rng.standard_normal((n, d))).astype(dtype)


def _boxes(X, k, b, seed):
    rng = np.random.default_rng(seed)
    c = X[rng.integers(0, len(X), (b, k))]
    h = np.exp(rng.uniform(np.log(1e-3), np.log(4), (b, k, X.shape[1]))) * (np.ptp(X, 0) / 20)
    return (c - h).astype(X.dtype), (c + h).astype(X.dtype)


def _check_bounds(X, k, lo, hi):
    kc = KCenter(_t(X), k)
    lb, raw, arg = (v.cpu().numpy() for v in kc.lower_bounds(_t(lo), _t(hi)))
    ref, refarg = oracle.lower_bounds(X, lo, hi)
    np.testing.assert_array_equal(raw, ref)
    np.testing.assert_array_equal(arg, refarg)
    assert np.all(lb <= ref) and np.all(lb >= ref * (1 - 1e-13))
    kc.close()


def _check_sets(X, k, sets):
    kc = KCenter(_t(X), k)
    for _ in range(2):   # the second call finds the workspace as the first left it
        ub, worst = (v.cpu().numpy() for v in kc.upper_bound(_t(sets)))
        for i in range(len(sets)):
            v, w = oracle.objective(X, sets[i])
            assert ub[i] == v and worst[i] == w, i
    kc.close()


@pytest.mark.parametrize("n,d,k,b", [(300, 2, 3, 1), (4_097, 1, 2, 9), (60_001, 4, 3, 70), (9_001, 7, 5, 130),
                                     (5_003, 13, 7, 64), (3_001, 29, 3, 65), (2_500, 68, 4, 33), (1_300, 128, 3, 17),
                                     (700_001, 3, 2, 3)])
def test_double_bounds(n, d, k, b):
    X = _data(n, d, k, n + d, np.float64)
    _check_bounds(X, k, *_boxes(X, k, b, d))


@pytest.mark.parametrize("shift,scale", [(1e6, 1.0), (-3e9, 1e-3), (0.0, 1e16), (0.0, 1e-20), (0.0, 1e140)])
def test_double_bounds_offset_and_range(shift, scale):
    X = (shift + _data(40_003, 3, 3, 5, np.float64)) * scale
    lo, hi = _boxes(X, 3, 40, 7)
    lo[1], hi[1] = X[:3], X[:3]
    _check_bounds(X, 3, lo, hi)


def test_double_maxima_closer_than_float():
    """Many samples whose values differ by a few units in the last place of a
    double: the screen keeps them all, the smallest exact winner is found."""
    X = _data(50_000, 3, 2, 9, np.float64)
    far = X[0] + 100
    rng = np.random.default_rng(1)
    X[1::7] = far * (1 + rng.integers(-8, 9, (len(X[1::7]), 1)) * 2.0 ** -52)
    lo, hi = _boxes(X[2:40:7], 2, 30, 3)
    _check_bounds(X, 2, lo, hi)
    _check_bounds(np.tile(X[:50], (900, 1)), 2, lo, hi)
    lo[::4], hi[::4] = -1e3, 1e3   # bound 0 at sample 0
    _check_bounds(X, 2, lo, hi)


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("n,d,k,s", [(257, 2, 3, 1), (127, 1, 1, 5), (100_003, 4, 3, 2), (20_001, 8, 5, 9),
                                     (30_011, 3, 4, 300), (5_001, 16, 16, 20), (4_001, 29, 2, 40), (900, 128, 3, 7),
                                     (2_049, 5, 2, 64)])
def test_objectives(dtype, n, d, k, s):
    X = _data(n, d, k, n, dtype)
    rng = np.random.default_rng(s)
    near = np.argsort(((X - X[0]) ** 2).sum(1))[:64]
    sets = rng.integers(0, n, (s, k))
    sets[: s // 2, 0] = rng.choice(near, s // 2)   # similar sets
    _check_sets(X, k, sets)


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
def test_objective_ties(dtype):
    X = np.sign(_data(9_001, 3, 3, 3, dtype) - 10)
    _check_sets(X, 3, np.random.default_rng(0).integers(0, 9_001, (20, 3)))
    _check_sets(np.ones_like(X), 2, np.random.default_rng(0).integers(0, 9_001, (5, 2)))


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("s", [1, 3, 100])
def test_farthest_first_repeats(dtype, s):
    """Every call on one context gives the oracle's traversal."""
    X = _data(20_003, 3, 4, 8, dtype)
    kc = KCenter(_t(X), 4)
    starts = np.random.default_rng(s).integers(0, len(X), s)
    for _ in range(3):
        c, obj = (v.cpu().numpy() for v in kc.fft_multi(_t(starts)))
        for i in range(0, s, 9):
            rc, robj = oracle.fft(X, 4, int(starts[i]))
            assert np.array_equal(c[i], rc) and obj[i] == robj
    kc.close()
