"""A pivot that is not finite is reported as NOT_SPD at every basis size, on either side of the solve
classes, in every column of an 8 x 8 diagonal block, without and with refinement, and when the
adjoint refactors: an infinite mask entry, and finite ones whose product with lambda overflows."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

NOT_SPD = 4
SIZES = [50, 64, 100, 101, 104, 120, 128, 129, 150, 200, 201, 208, 209, 250, 304]
ROWS = 9


def _batch(kx, lam, ir):
    from paper_2604_10377_gb300 import api
    rng = np.random.default_rng(kx)
    d = 16 * ((2 * kx + 15) // 16)
    lay = api.BatchLayout([8, 8], [kx, ROWS], [d, d], "fp32")
    b = api.FmapBatch(lay, [(0, 1, lam)], with_grad=False, masks=[rng.uniform(0.5, 50.0, (ROWS, kx))], ir_steps=ir,
                      adjoint_ir_steps=ir)
    b.A.copy_(torch.from_numpy((0.05 * rng.standard_normal(b.A.numel())).astype(np.float32)))
    return b


@pytest.mark.parametrize("value,lam", [(np.inf, 1e-2), (3e38, 10.0)])
@pytest.mark.parametrize("ir", [0, 1])
@pytest.mark.parametrize("kx", SIZES)
def test_infinite_pivot_is_reported(kx, ir, value, lam):
    b = _batch(kx, lam, ir)
    mask = b.mask.view(ROWS, kx)
    clean = b.solve().clone()
    assert int(b.status[0]) == 0
    dc = torch.ones_like(clean)
    da = b.adjoint(dc, c=clean, use_saved=False).clone()
    assert int(b.status[0]) == 0 and bool(torch.isfinite(da).all())
    for j in sorted({0, 3, 6, 7, 8 * (kx // 16) + 5, kx - 2, kx - 1}):
        keep = float(mask[4, j])
        mask[4, j] = value
        c = b.c_view(b.solve(c_out=torch.empty_like(clean)), 0).cpu().numpy()
        assert int(b.status[0]) == (NOT_SPD | (4 << 8)), j
        assert np.all(np.isnan(c[4])) and np.array_equal(np.delete(c, 4, 0), np.delete(b.c_view(clean, 0).cpu().numpy(), 4, 0))
        b.status.zero_()
        b.adjoint(dc, c=clean, use_saved=False)
        assert int(b.status[0]) == (NOT_SPD | (4 << 8)), j
        mask[4, j] = keep
        b.status.zero_()
