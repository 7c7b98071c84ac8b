"""Many center sets at once: any number is taken (a launch's node ranges are
bounded), and the screen's tile maxima stay within 256 MiB whatever the tile."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2301_00061_gb300 import KCenter  # noqa: E402

DEV = torch.device("cuda:0")


def _sets(s, k, n, seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    return torch.randint(0, n, (s, k), generator=g, device=DEV)


def test_more_sets_than_a_grid_has_ranges():
    """At K = 16, D = 128 about six nodes fit a CTA: 400,000 sets are more than
    65,535 ranges."""
    n, d, k, s = 1_000, 128, 16, 400_000
    X = np.random.default_rng(0).normal(size=(n, d)).astype(np.float32)
    sets = _sets(s, k, n, 1)
    with KCenter(torch.from_numpy(X).to(DEV), k) as kc:
        ub, worst = kc.upper_bound(sets)
        for lo in (0, s - 1_000):
            u, w = kc.upper_bound(sets[lo:lo + 1_000].contiguous())
            assert torch.equal(u, ub[lo:lo + 1_000]) and torch.equal(w, worst[lo:lo + 1_000])
    for i in (0, 65_535, 65_536, 262_143, s - 1):
        v, w = oracle.objective(X, sets[i].cpu().numpy())
        assert float(ub[i]) == v and int(worst[i]) == w


# tiles of 128 samples: wide data (pruning kernel), and few sets at D <= 8 (streaming)
@pytest.mark.parametrize("n,d,k,s", [(400_000, 70, 1, 40_000), (60_000_000, 1, 1, 200)])
def test_screen_workspace(n, d, k, s):
    g = torch.Generator(device=DEV)
    g.manual_seed(2)
    X = torch.randn(n, d, generator=g, device=DEV)
    sets = _sets(s, k, n, 3)
    ub, worst = torch.empty(s, dtype=torch.float64, device=DEV), torch.empty(s, dtype=torch.int64, device=DEV)
    import paper_2301_00061_gb300 as kcm
    with KCenter(X, k) as kc:
        kc.upper_bound(sets[:1].contiguous())
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        kcm.kc_upper_bound(kc.h, sets, ub, worst)
        torch.cuda.synchronize()
        held = free - torch.cuda.mem_get_info()[0]
    assert held < (320 << 20), held
    # the values, by the definition in 64 bits
    for i in (0, s // 2, s - 1):
        far = (X.double() - X[sets[i, 0]].double()).square().sum(1)
        assert abs(float(ub[i]) - float(far.max())) <= 1e-12 * float(ub[i]) and float(far[worst[i]]) >= float(far.max()) * (1 - 1e-12)
