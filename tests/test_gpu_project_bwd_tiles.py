"""Backward projection from given dL/dA at the edges of its tiles: vertex counts around the 128- and
256-vertex tiles, features around the 16-, 32- and 64-column pieces and the 256-feature groups,
basis sizes from one 32-column block to ten, shapes of different sizes in one batch (each work
item divides the shared memory by its own basis size). Against FP64; TF32 operands give about
6e-4 (BF16 batches, the FP32 copy: 1e-3), BF16 storage 3e-3, the three FP32 passes 1e-5."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _check(ns, ks, ds, feat, **kw):
    from paper_2604_10377_gb300 import api
    rng = np.random.default_rng(sum(ns) + sum(ks))
    lay = api.BatchLayout(ns, ks, ds, feat)
    b = api.FmapBatch(lay, [(0, 0, 1e-2)], precision=feat, with_grad=True, grad_f32_copy=feat == "bf16", **kw)
    b.dfeat.fill_(7.0)
    refs = []
    for s, (n, k, d) in enumerate(zip(ns, ks, ds)):
        phi, mass = rng.standard_normal((n, k)).astype(np.float32), rng.uniform(0.5, 1.5, n).astype(np.float32)
        da = rng.standard_normal((k, d)).astype(np.float32)
        b.phi[lay.phi_off[s]:lay.phi_off[s] + n * lay.ld_phi[s]].view(n, -1)[:, :k] = torch.from_numpy(phi).cuda()
        b.mass[lay.mass_off[s]:lay.mass_off[s] + n] = torch.from_numpy(mass).cuda()
        b.a_view(b.dA, s).copy_(torch.from_numpy(da))
        refs.append(mass[:, None].astype(np.float64) * (phi.astype(np.float64) @ da.astype(np.float64)))
    b.project_backward()
    assert int(b.status[0]) == 0
    used = torch.zeros(b.dfeat.numel(), dtype=torch.bool, device="cuda")
    for s, ref in enumerate(refs):
        used[lay.feat_off[s]:lay.feat_off[s] + ref.size] = True

        def rel(flat):
            return np.linalg.norm(lay.feat_view(flat, s).double().cpu().numpy() - ref) / np.linalg.norm(ref)
        assert rel(b.dfeat) <= (3e-3 if feat == "bf16" else 1e-5)
        if feat == "bf16":
            assert rel(b.dfeat32) <= 1e-3
    assert bool((b.dfeat[~used] == 7.0).all())      # nothing outside the shapes' rows


@pytest.mark.parametrize("feat", ["bf16", "fp32"])
@pytest.mark.parametrize("d", [16, 48, 80, 256, 272, 528])
def test_vertex_and_feature_edges(d, feat):
    ns = [1, 31, 127, 128, 129, 255, 256, 257, 1023, 1025, 2300]
    _check(ns, [7 if n % 2 else 40 for n in ns], [d] * len(ns), feat)


@pytest.mark.parametrize("feat", ["bf16", "fp32"])
@pytest.mark.parametrize("kw", [{}, {"tuning": {"bwd_ctas": 4}}, {"tuning": {"bwd_group_features": 64, "bwd_chunk_v": 1152}}])
def test_mixed_basis_sizes(feat, kw):
    ks = [1, 32, 33, 64, 100, 128, 160, 200, 224, 256, 300, 304]
    _check([3000 + 17 * k for k in ks], ks, [144 if k % 3 else 320 for k in ks], feat, **kw)
