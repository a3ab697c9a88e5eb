"""Gram matrix and right-hand sides at the edges of their 32 x 32 tiles and of the slabs of 16
features that a block's thread groups share (fewer slabs than groups, remainders), FP32 and
double-float sums, maps with other row counts, and descriptors off the 16-byte alignment:
through the map C, against 64-bit linear algebra."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from test_gpu_row_solve_classes import CTOL, _batch, _reference, _rel  # noqa: E402


@pytest.mark.parametrize("hi_min", [1, 1000])
@pytest.mark.parametrize("kxs,ky,d", [((1, 7), 3, 16), ((15, 16), 33, 48), ((31, 32, 33), 31, 80), ((63, 65), 64, 144),
                                      ((97, 130), 32, 272), ((200,), 65, 400), ((200, 160) * 24, 5, 400)])
def test_map_through_the_gram_matrix(kxs, ky, d, hi_min):
    lam = float(np.float32(1e-2))
    b, a, ev, _, dc = _batch(kxs, ky, d, 0.05, hi_gram_min_k=hi_min)
    c = b.solve()
    shifted = torch.zeros(b.A.numel() + 1, device="cuda")[1:]      # 4-byte aligned descriptors
    shifted.copy_(b.A)
    c1 = b.solve(shifted, c_out=torch.empty_like(c))
    assert torch.equal(c, c1)
    assert int(b.status[:len(kxs)].abs().sum()) == 0
    for p in range(min(len(kxs), 4)):
        rc, _, _ = _reference(a[2 * p], a[2 * p + 1], ev[2 * p], ev[2 * p + 1], None, lam, dc[p])
        assert _rel(b.c_view(c, p).cpu().numpy(), rc) <= CTOL
