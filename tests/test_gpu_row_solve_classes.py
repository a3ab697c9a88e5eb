"""Row systems at the edges of the solve classes (k_X = 64 | 100 | 128 | 200 | 208 | 304) and of
their 8-column panels and 16-row blocks, from given descriptors: the map, the adjoint with saved
and with recomputed factors, a system that is not positive definite and one whose pivots are
subnormal, against 64-bit linear algebra. Few rows per map: a row is one system."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

CTOL, GTOL = 1e-5, 1e-4     # FP32 mode: C, gradients (as in the parity tests)
EDGES = [(63, 64, 65), (96, 99, 100, 101, 104), (105, 112, 127, 128, 129), (136, 137, 144, 153), (199, 200, 201),
         (207, 208, 209), (255, 256, 264), (297, 303, 304)]


def _batch(kxs, ky, d, scale, with_mask=False, **kw):
    from paper_2604_10377_gb300 import api
    rng = np.random.default_rng(sum(kxs) + ky)
    ks = [k for kx in kxs for k in (kx, ky)]
    lay = api.BatchLayout([8] * len(ks), ks, [d] * len(ks), "fp32")
    masks = [rng.uniform(0.5, 50.0, (ky, kx)).astype(np.float32) for kx in kxs] if with_mask else None
    b = api.FmapBatch(lay, [(2 * p, 2 * p + 1, 1e-2) for p in range(len(kxs))], with_grad=False, masks=masks, **kw)
    a = [(scale * rng.standard_normal((k, d))).astype(np.float32) for k in ks]
    ev = [np.sort(rng.uniform(0, 10, k)).astype(np.float32) for k in ks]
    for s, k in enumerate(ks):
        b.a_view(b.A, s).copy_(torch.from_numpy(a[s]))
        b.evals[lay.evals_off[s]:lay.evals_off[s] + k] = torch.from_numpy(ev[s]).cuda()
    dc = [rng.standard_normal((ky, kx)).astype(np.float32) for kx in kxs]
    return b, a, ev, masks, dc


def _reference(ax, ay, evx, evy, mask, lam, dc):
    ax, ay = ax.astype(np.float64), ay.astype(np.float64)
    dm = mask.astype(np.float64) if mask is not None else (evy.astype(np.float64)[:, None] - evx[None].astype(np.float64)) ** 2
    g, r = ax @ ax.T, ay @ ax.T
    c, gam = np.empty_like(r), np.empty_like(r)
    for i in range(r.shape[0]):
        c[i], gam[i] = np.linalg.solve(g + lam * np.diag(dm[i]), np.stack([r[i], dc[i]], 1)).T
    return c, gam.T @ ay - (gam.T @ c + c.T @ gam) @ ax, gam @ ax


def _rel(x, ref):
    return np.linalg.norm(np.asarray(x, np.float64) - ref) / np.linalg.norm(ref)


@pytest.mark.parametrize("use_saved", [True, False])
@pytest.mark.parametrize("kxs", EDGES)
def test_map_and_adjoint(kxs, use_saved):
    lam = float(np.float32(1e-2))
    b, a, ev, masks, dc = _batch(kxs, 9, 16 * ((2 * max(kxs) + 15) // 16), 0.05, with_mask=min(kxs) % 2 == 1)
    from paper_2604_10377_gb300 import api
    c = b.solve()
    da = b.adjoint(api.flat_c(b, dc), use_saved=use_saved)
    assert int(b.status[:len(kxs)].abs().sum()) == 0
    for p in range(len(kxs)):
        rc, gx, gy = _reference(a[2 * p], a[2 * p + 1], ev[2 * p], ev[2 * p + 1], masks[p] if masks else None, lam, dc[p])
        assert _rel(b.c_view(c, p).cpu().numpy(), rc) <= CTOL
        assert _rel(b.a_view(da, 2 * p).cpu().numpy(), gx) <= GTOL
        assert _rel(b.a_view(da, 2 * p + 1).cpu().numpy(), gy) <= GTOL


@pytest.mark.parametrize("kx", [64, 100, 104, 128, 150, 200, 208, 250])
def test_bad_pivot_is_reported(kx):
    b, a, ev, masks, dc = _batch((kx,), 9, 512, 0.05, with_mask=True)
    m = b.mask.view(9, kx)
    m[4, kx - 2] = -1e9
    c = b.solve()
    assert int(b.status[0]) == (4 | (4 << 8))
    c = b.c_view(c, 0).cpu().numpy()
    assert np.all(np.isnan(c[4])) and np.all(np.isfinite(np.delete(c, 4, axis=0)))


@pytest.mark.parametrize("kx", [50, 100, 104, 128, 150, 250])
def test_subnormal_pivots_are_accepted(kx):
    """G of about 3e-39 (below the smallest normal FP32 number): products keep about 1e-4 of
    relative precision there and sums of 512 more, so C is right to a few percent."""
    b, a, ev, masks, dc = _batch((kx,), 9, 512, 2.0 ** -68.5, hi_gram_min_k=1000, ir_steps=0)
    b.evals.zero_()
    c = b.solve()
    assert int(b.status[0]) == 0
    rc, _, _ = _reference(a[0], a[1], 0 * ev[0], 0 * ev[1], None, 0.0, dc[0])
    assert _rel(b.c_view(c, 0).cpu().numpy(), rc) <= 5e-2
