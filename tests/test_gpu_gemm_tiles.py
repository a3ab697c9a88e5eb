"""Training loss and adjoint GEMMs on the CUDA cores, on 64 x 64 and 32 x 32 output tiles: batches on
either side of the line between them, basis sizes and features around the tiles' edges and the slabs of 16
reduction indices, square and rectangular maps, every pair's loss and dL/dC and every shape's dL/dA.
Against FP64: FP32 sums of up to 608 products, 1e-5; dL/dA as in the parity tests, 1e-4."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from test_gpu_row_solve_classes import GTOL, _reference, _rel  # noqa: E402


def _tiles(pairs, ks, d, t):
    up = lambda n: -(-n // t)  # noqa: E731
    loss = sum(up(ks[y]) * up(max(ks[x], ks[y])) for x, y in pairs)
    return loss, sum((up(ks[x]) + up(ks[y])) * up(d) for x, y in pairs)


@pytest.mark.parametrize("ks,d,n_pairs,tile", [((64, 64, 61), 144, 240, 64), ((100, 128, 97), 144, 70, 64),
                                               ((128, 127, 100), 272, 64, 64), ((250, 239), 512, 20, 64),
                                               ((100, 128, 97), 144, 20, 32), ((65, 33, 90), 80, 130, 32),
                                               ((8, 1, 17), 16, 40, 32), ((304, 290), 608, 2, 32)])
def test_loss_and_adjoint_tiles(ks, d, n_pairs, tile):
    from paper_2604_10377_gb300 import api
    n = len(ks)
    pairs = [(p % n, (p // n) % n) for p in range(n_pairs)]
    l32, a32 = _tiles(pairs, ks, d, 32)
    l64, a64 = _tiles(pairs, ks, d, 64)
    assert ((l32 > 912 and l32 > 3.2 * l64) or (a32 > 2280 and a32 > 3.5 * a64)) == (tile == 64)
    rng = np.random.default_rng(sum(ks))
    lay = api.BatchLayout([8] * n, ks, [d] * n, "fp32")
    b = api.FmapBatch(lay, [(x, y, 1e-2) for x, y in pairs], with_grad=False, tuning={"adjoint_kernel": 2})
    a = [(0.05 * rng.standard_normal((k, d))).astype(np.float32) for k in ks]
    ev = [np.sort(rng.uniform(0, 10, k)).astype(np.float32) for k in ks]
    for s, k in enumerate(ks):
        b.a_view(b.A, s).copy_(torch.from_numpy(a[s]))
        b.evals[lay.evals_off[s]:lay.evals_off[s] + k] = torch.from_numpy(ev[s]).cuda()
    c = b.solve()
    gt = [rng.standard_normal((ks[y], ks[x])).astype(np.float32) for x, y in pairs]
    loss, dc = b.loss_orth(c, api.flat_c(b, gt))
    dcs = [rng.standard_normal(g.shape).astype(np.float32) for g in gt]
    da = b.adjoint(api.flat_c(b, dcs))
    assert int(b.status.abs().sum()) == 0
    want = [np.zeros((k, d)) for k in ks]
    lam = float(np.float32(1e-2))
    loss = loss.cpu().numpy().astype(np.float64)
    for p, (x, y) in enumerate(pairs):
        cp = b.c_view(c, p).cpu().numpy().astype(np.float64)
        e, r = cp @ cp.T - np.eye(ks[y]), cp - gt[p]
        assert abs(loss[p] - (e ** 2).sum() - (r ** 2).sum()) <= 1e-5 * loss[p]
        assert _rel(b.c_view(dc, p).cpu().numpy(), 4 * e @ cp + 2 * r) <= 1e-5
        _, gx, gy = _reference(a[x], a[y], ev[x], ev[y], None, lam, dcs[p])
        want[x] += gx
        want[y] += gy
    for s in {s for q in pairs for s in q}:
        assert _rel(b.a_view(da, s).cpu().numpy(), want[s]) <= GTOL
