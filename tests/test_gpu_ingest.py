"""Loading a dataset: device, pinned and pageable rows give the same bounds and
root box, at tile edges of the transpose (24 KB of rows, a multiple of 16) and of the
root box's 16-byte groups, from an address that is not 16-byte aligned too."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
import paper_2301_00061_gb300 as kcm  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("n,d", [(1, 1), (2, 3), (63, 8), (768, 8), (769, 8), (3073, 2), (80, 68), (16, 128), (17, 128),
                                 (100_003, 5)])
def test_rows_from_anywhere(n, d, dtype):
    g = torch.Generator().manual_seed(n * 131 + d)
    flat = torch.randn(n * d + 1, generator=g, dtype=torch.float64).to(dtype)
    flat[n * d // 2] = -0.0
    for off in (0, 1):   # (1: element-aligned only)
        X = flat[off:off + n * d].reshape(n, d)
        pinned = flat.pin_memory()[off:off + n * d].reshape(n, d)
        device = flat.cuda()[off:off + n * d].reshape(n, d)
        lo, hi = X.min(0).values.double().numpy(), X.max(0).values.double().numpy()
        box = np.stack([np.stack([lo]), np.stack([lo])])   # two nodes: the corner point
        want = None
        for rows in (X, pinned, device):
            with kcm.KCenter(rows, 1) as kc:
                rlo, rhi = kc.root_box()
                assert np.array_equal(np.asarray(torch.as_tensor(rlo).cpu(), dtype=np.float64).ravel(), lo)
                assert np.array_equal(np.asarray(torch.as_tensor(rhi).cpu(), dtype=np.float64).ravel(), hi)
                t = torch.as_tensor(box).to(dtype).cuda()
                got = [np.asarray(torch.as_tensor(o).cpu()) for o in kc.lower_bounds(t, t)]
            if want is None:
                want = got
            for a, b in zip(want, got):
                assert np.array_equal(a, b)
