"""Spatial gradient features where the gather's bookkeeping can go wrong: rows of 0, 1, 7, 8, 9 and
40 entries side by side, neighbours far outside a tile, tiles of one vertex, K-blocks from one to
eight, and infinities in rows of X that no entry names. Against FP64 products; TF32 operands give
about 6e-4, the FP32 tolerance of the feature tests is 1.5e-3."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,dim", [(1, 16), (128, 48), (129, 112), (700, 128), (20000, 32), (40000, 128)])
@pytest.mark.parametrize("variant", ["A", "B"])
def test_uneven_rows(n, dim, variant):
    from paper_2604_10377_gb300 import api
    rng = np.random.default_rng(n + dim)
    lens = np.array([0, 1, 7, 8, 9, 40])[rng.integers(0, 6, n)]
    lens[-1] = 7
    n_in = n + 5
    ptr = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    nnz = int(ptr[-1])
    col = rng.integers(0, n, nnz).astype(np.int32)          # rows n .. n + 4 of X are never named
    vals = (rng.standard_normal((nnz, 2)) / 4).astype(np.float32)
    x = np.full((n_in, dim + 4), np.inf, np.float32)        # nor are the columns past dim
    x[:n, :dim] = rng.standard_normal((n, dim))
    ar, ai = (rng.standard_normal((2, dim, dim)) / np.sqrt(dim)).astype(np.float32)
    out, status = api.gradient_features(*(torch.from_numpy(t).cuda() for t in (ptr, col, vals, x)),
                                        torch.from_numpy(ar).cuda(), torch.from_numpy(ai).cuda(), variant=variant)
    assert int(status) == 0
    row = np.repeat(np.arange(n), lens)
    zx, zy = np.zeros((n, dim)), np.zeros((n, dim))
    np.add.at(zx, row, vals[:, :1].astype(np.float64) * x[col, :dim])
    np.add.at(zy, row, vals[:, 1:].astype(np.float64) * x[col, :dim])
    p = zx @ ar.T.astype(np.float64) - zy @ ai.T
    q = (zy @ ar.T.astype(np.float64) + zx @ ai.T) if variant == "A" else (zx @ ar.T.astype(np.float64) + zy @ ai.T)
    ref = zx * p + zy * q
    got = out.cpu().numpy().astype(np.float64)
    assert np.linalg.norm(got - ref) <= 1.5e-3 * np.linalg.norm(ref)
    assert np.all(got[lens == 0] == 0)
