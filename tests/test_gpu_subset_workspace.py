"""Batches of nodes over a long list of ids: the rows are gathered a part at a time,
within a bounded workspace, and the parts join at the same value and sample."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2301_00061_gb300 as kcm  # noqa: E402
from paper_2301_00061_gb300 import KCenter  # noqa: E402

DEV = torch.device("cuda:0")


@pytest.mark.parametrize("n,d,k,b", [(9_000_001, 8, 2, 40), (20_000_000, 3, 3, 70)])
@pytest.mark.parametrize("spread", [1000, 3])   # few equal values; many
def test_long_lists(n, d, k, b, spread):
    g = torch.Generator(device=DEV)
    g.manual_seed(n + spread)
    X = torch.randint(0, spread, (n, d), generator=g, device=DEV).float()
    lo = torch.randint(0, spread, (b, k, d), generator=g, device=DEV).float()
    hi = lo + torch.randint(0, spread, (b, k, d), generator=g, device=DEV).float()
    ids = torch.arange(n, device=DEV, dtype=torch.int32).flip(0).contiguous()
    out = [torch.empty(b, dtype=torch.float64, device=DEV) for _ in range(2)]
    arg = torch.empty(b, dtype=torch.int64, device=DEV)
    with KCenter(X, k) as kc:
        want = kc.lower_bounds(lo, hi)
        kcm.kc_lower_bounds_subset(kc.h, ids[:1000], lo, hi, out[0], out[1], arg)
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        kcm.kc_lower_bounds_subset(kc.h, ids, lo, hi, out[0], out[1], arg)
        torch.cuda.synchronize()
        held = free - torch.cuda.mem_get_info()[0]
    assert held < (160 << 20), held
    for a, w in zip((out[0], out[1], arg), want):
        assert torch.equal(a, w)
