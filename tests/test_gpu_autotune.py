"""The launch shapes that kc_autotune tries and keeps: bounds stay bit for bit those
of the untuned context, for the tuned batch and for others after it; a batch that is
evaluated in full leaves nothing behind."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2301_00061_gb300 as kcm  # noqa: E402
from paper_2301_00061_gb300 import KCenter  # noqa: E402

DEV = torch.device("cuda:0")


def _boxes(X, k, b, seed):
    rng = np.random.default_rng(seed)
    c = X[rng.integers(0, len(X), k)]
    h = np.sort(rng.uniform(0, 3, (b, k, 1)), 0)[::-1] + np.zeros((1, 1, X.shape[1]))
    return [torch.from_numpy(np.ascontiguousarray(v.astype(np.float32))).to(DEV) for v in (c - h, c + h)]


@pytest.mark.parametrize("n,d,k,b", [(300_001, 8, 5, 77), (1_000_003, 3, 3, 130), (200_000, 12, 4, 33), (60_000, 29, 3, 9)])
def test_tuned_bounds_are_the_untuned(n, d, k, b):
    X = np.random.default_rng(d).normal(size=(n, d)).astype(np.float32)
    Xd = torch.from_numpy(X).to(DEV)
    batches = [_boxes(X, k, q, q) for q in (b, 1, 9, 300)]
    with KCenter(Xd, k) as kc, KCenter(Xd, k) as plain:
        st, chunk, ms = kcm.kc_autotune(kc.h, *batches[0])
        assert st in (1, 2, 4) and (chunk == b or (chunk < b and chunk % 8 == 0)) and ms > 0
        for lo, hi in batches:
            for a, w in zip(kc.lower_bounds(lo, hi), plain.lower_bounds(lo, hi)):
                assert torch.equal(a, w)


def test_batches_evaluated_in_full_have_nothing_to_tune():
    X = np.random.default_rng(1).normal(size=(300_000, 4)).astype(np.float32)
    with KCenter(torch.from_numpy(X).to(DEV), 3) as kc:
        st, chunk, ms = kcm.kc_autotune(kc.h, *_boxes(X, 3, 4, 1))
        assert st == 0 and chunk == 0 and ms > 0
