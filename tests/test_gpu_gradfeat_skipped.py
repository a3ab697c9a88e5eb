"""Entries of the gradient operator whose column is out of range are skipped, whatever their values: the
status reports them and the features are those of the operator without them."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("value", [np.inf, np.nan, 3e38])
@pytest.mark.parametrize("per_row", [3, 8, 20])
def test_skipped_entries_leave_no_trace(per_row, value):
    from paper_2604_10377_gb300 import api
    n, dim = 300, 32
    rng = np.random.default_rng(per_row)
    ptr = (per_row * np.arange(n + 1)).astype(np.int64)
    col = rng.integers(0, n, n * per_row).astype(np.int32)
    vals = rng.standard_normal((n * per_row, 2)).astype(np.float32)
    x, ar, ai = (torch.from_numpy(rng.standard_normal(s).astype(np.float32)).cuda() for s in ((n, dim), (dim, dim), (dim, dim)))
    bad = rng.choice(n * per_row, 40, replace=False)

    def run(c, v):
        out, status = api.gradient_features(torch.from_numpy(ptr).cuda(), torch.from_numpy(c).cuda(),
                                            torch.from_numpy(v).cuda(), x, ar, ai)
        return out, int(status)
    v0 = vals.copy()
    v0[bad] = 0.0                                       # in range, without weight
    want, status = run(col, v0)
    assert status == 0
    c1, v1 = col.copy(), vals.copy()
    c1[bad[::2]], c1[bad[1::2]] = n, -1
    v1[bad] = value
    got, status = run(c1, v1)
    assert status == 1
    assert torch.equal(got, want)
