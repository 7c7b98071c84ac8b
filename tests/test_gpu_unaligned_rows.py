"""Pinned host rows at an address that is no multiple of their element size: a
kernel cannot read them where they are, so they are copied first, as pageable rows
are."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2301_00061_gb300 import KCenter  # noqa: E402


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("off", [1, 2, 3, 4, 8, 12])
@pytest.mark.parametrize("n,d", [(1_000, 1), (5_003, 3), (4_096, 8)])
def test_pinned_rows_at_any_address(dtype, off, n, d):
    X = np.random.default_rng(off).normal(size=(n, d)).astype(dtype)
    raw = torch.empty(X.nbytes + 64, dtype=torch.uint8).pin_memory()
    rows = raw.numpy()[off:off + X.nbytes].view(dtype).reshape(n, d)
    assert rows.ctypes.data == raw.data_ptr() + off
    rows[:] = X
    with KCenter(rows, 2) as kc:
        lo, hi = kc.root_box()
        sets = np.array([[0, n - 1], [n // 2, 1]], np.int64)
        ub, worst = kc.upper_bound(sets)
    np.testing.assert_array_equal(lo, X.min(0))
    np.testing.assert_array_equal(hi, X.max(0))
    for i in range(2):
        v, w = oracle.objective(X, sets[i])
        assert ub[i] == v and worst[i] == w
