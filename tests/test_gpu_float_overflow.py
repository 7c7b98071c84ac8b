"""Finite float data so far apart that squared distances leave the float range:
every value still equals the FP64 oracle, every certified bound stays at or
below it, and farthest-first traversal names samples.  Scaling by a power of two
changes no rounding in double, so the unscaled data give the expected values."""
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


# 2^60: distances straddle the float range; 2^66: every one leaves it
SHAPES = [(3_001, 2, 3, 60), (20_001, 5, 2, 66), (2_500, 29, 3, 66), (700, 128, 2, 60), (60_000, 3, 4, 64)]


def _data(n, d, k, e):
    rng = np.random.default_rng(n + d)
    means = rng.uniform(-20, 20, (k, d))
    X = (means[rng.integers(0, k, n)] + rng.standard_normal((n, d))).astype(np.float32)
    return X * np.float32(2.0) ** np.float32(e)


@pytest.mark.parametrize("n,d,k,e", SHAPES)
@pytest.mark.parametrize("s", [1, 40])
def test_objectives(n, d, k, e, s):
    X = _data(n, d, k, e)
    rng = np.random.default_rng(s)
    sets = rng.integers(0, n, (s, k))
    pts = (X[sets] * np.float32(1.5)).astype(np.float32)
    with KCenter(_t(X), k) as kc:
        ub, worst = (v.cpu().numpy() for v in kc.upper_bound(_t(sets)))
        up, wp = (v.cpu().numpy() for v in kc.upper_bound_points(_t(pts)))
    # (the same objective as an oracle of points: the lower bound of point boxes)
    refp, refpw = oracle.lower_bounds(X, pts, pts)
    for i in range(s):
        v, w = oracle.objective(X, sets[i])
        assert np.isfinite(v) and ub[i] == v and worst[i] == w
    np.testing.assert_array_equal(up, refp)
    np.testing.assert_array_equal(wp, refpw)


@pytest.mark.parametrize("n,d,k,e", SHAPES)
def test_farthest_first(n, d, k, e):
    X = _data(n, d, k, e)
    with KCenter(_t(X), k) as kc:
        starts = np.array([0, n // 2, n - 1])
        cs, obj = (v.cpu().numpy() for v in kc.fft_multi(_t(starts)))
        for i, st in enumerate(starts):
            assert cs[i, 0] == st and np.all(cs[i] >= 0) and np.all(cs[i] < n)
            for t in range(1, k):
                assert cs[i, t] == oracle.objective(X, cs[i, :t])[1]
            assert obj[i] == oracle.objective(X, cs[i])[0]
            one, val = kc.fft(int(st))
            np.testing.assert_array_equal(np.asarray(one), cs[i])
            assert val[0] == obj[i]


@pytest.mark.parametrize("n,d,k,e", SHAPES)
@pytest.mark.parametrize("b", [2, 70])
def test_bounds_stay_below(n, d, k, e, b):
    X = _data(n, d, k, e)
    rng = np.random.default_rng(b)
    c = X[rng.integers(0, n, (b, k))]
    h = rng.uniform(0, 0.2, (b, k, d)).astype(np.float32) * np.ptp(X, 0)
    lo, hi = c - h, c + h
    ref, _ = oracle.lower_bounds(X, lo, hi)
    top = float(np.finfo(np.float32).max)
    with KCenter(_t(X), k) as kc:
        lb = kc.lower_bounds(_t(lo), _t(hi))[0].cpu().numpy()
        t = kc.tighten(_t(lo), _t(hi), top)["lb"].cpu().numpy()
        lists = [lb, t]
        if d <= 8:
            ids = np.arange(n, dtype=np.int32)
            lists.append(kc.lower_bounds_subset(_t(ids), _t(lo), _t(hi))[0].cpu().numpy())
    for v in lists:
        assert np.all(np.isfinite(v)) and np.all(v <= ref)
        # as tight as the float evaluation allows, up to the float range's end
        assert np.all(v >= np.minimum(ref, top) * (1 - 2e-5))


def test_double_bounds_beyond_the_double_range():
    X = _data(300, 3, 2, 0).astype(np.float64) * 2.0 ** 700
    lo = np.repeat(X[:1, None], 2, 1)
    with KCenter(_t(X), 2) as kc:
        lb = kc.lower_bounds(_t(lo), _t(lo))[0].cpu().numpy()
    assert np.all(np.isfinite(lb)) and np.all(lb > 1.7e308)


@pytest.mark.parametrize("lists", [0, 1])
def test_solve(lists):
    """The optimum of the scaled data is the scaled optimum, and the certificate holds."""
    X = _data(60, 2, 2, 0)
    want = oracle.solve(X, 2, tol=1e-12)["objective"] * 2.0 ** 132
    with KCenter(_t(X * np.float32(2.0) ** np.float32(66)), 2) as kc:
        r = kc.solve(tol=1e-12, lists=lists, node_limit=20_000)
    assert r["lower_bound"] <= want * (1 + 1e-12)
    assert r["objective"] == oracle.objective(X, r["centers"])[0] * 2.0 ** 132
    if r["status"] == 0:
        assert abs(r["objective"] - want) <= 1e-12 * want
