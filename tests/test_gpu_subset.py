"""Bounds over a subset of the samples: the gathering stream (few nodes) and the
gathered batch against the FP64 oracle on the chosen rows, bit for bit on grid
data; the arg-max is the smallest sample index whatever the ids' order."""
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


@pytest.mark.parametrize("d", [1, 2, 3, 4, 5, 6, 7, 8])
@pytest.mark.parametrize("b", [1, 2, 9, 70])
def test_subset_any_order(d, b):
    rng = np.random.default_rng(10 * d + b)
    n, k = 5_003, 3
    means = rng.integers(-30, 30, (k, d))
    X = ((means[rng.integers(0, k, n)] + np.rint(4 * rng.standard_normal((n, d)))) / 4).astype(np.float32)
    at = means[None] / 4 + np.rint(rng.standard_normal((b, k, d)) * 4) / 4
    h = rng.integers(0, 16, (b, k, d)) / 4
    lo, hi = (at - h).astype(np.float32), (at + h).astype(np.float32)
    kc = KCenter(_t(X), k)
    for m, off in ((1, 0), (127, 1), (1_025, 3), (3_001, 0), (5_003, 2)):
        pool = np.concatenate([np.zeros(off, np.int64), rng.integers(0, n, m)]).astype(np.int32)
        ids = _t(pool)[off:]   # off elements past a 16-byte boundary, unsorted, repeated
        lb, raw, arg = (v.cpu().numpy() for v in kc.lower_bounds_subset(ids, _t(lo), _t(hi)))
        rows = np.unique(pool[off:])
        ref, at_ = oracle.lower_bounds(X[rows], lo, hi)
        np.testing.assert_array_equal(raw, ref)
        np.testing.assert_array_equal(arg, rows[at_])
        assert np.all(lb <= ref)
    kc.close()


def test_subset_of_everything_in_chunks():
    """33.6 million ids pass the gather buffer's chunk size: equal to the full bound."""
    n, d, k = (1 << 25) + 70_001, 2, 4
    g = torch.Generator(device=DEV)
    g.manual_seed(3)
    X = torch.randn(n, d, generator=g, device=DEV) + 8 * torch.randint(0, 3, (n, 1), generator=g, device=DEV)
    c = X[torch.randint(0, n, (40, k), generator=g, device=DEV)]
    lo, hi = (c - 0.5).contiguous(), (c + 0.5).contiguous()
    kc = KCenter(X, k)
    ids = torch.arange(n, dtype=torch.int32, device=DEV)
    for b in (2, 40):
        full = kc.lower_bounds(lo[:b].contiguous(), hi[:b].contiguous())
        part = kc.lower_bounds_subset(ids, lo[:b].contiguous(), hi[:b].contiguous())
        for u, v in zip(full, part):
            assert torch.equal(u, v)
    kc.close()
