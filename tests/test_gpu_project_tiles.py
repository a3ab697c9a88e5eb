"""Forward projection at the edges of its operand tiles and of its reduction: basis sizes around the
16-column MMA step and around those at which the head and remainder products run as one MMA (128
columns for two feature groups, fewer for three and four; three, two or one accumulators of the FP32
features' BF16 thirds: 64 and 96 columns for two groups, 80 for one), one vertex to more partials than the
reduction takes in one round. Against FP64: the BF16 features are exact, the basis is split into two
BF16 parts (2^-17 per product) and accumulated in FP32, 2e-5; FP32 features 2e-6."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _check(ns, ks, ds, feat, **kw):
    from paper_2604_10377_gb300 import api
    rng = np.random.default_rng(sum(ns) + sum(ks))
    lay = api.BatchLayout(ns, ks, ds, feat)
    b = api.FmapBatch(lay, [(0, 0, 1e-2)], precision=feat, **kw)
    refs = []
    for s, (n, k, d) in enumerate(zip(ns, ks, ds)):
        phi, mass = rng.standard_normal((n, k)).astype(np.float32), rng.uniform(0.5, 1.5, n).astype(np.float32)
        f = torch.from_numpy(rng.standard_normal((n, d)).astype(np.float32)).to(b.feat.dtype)
        b.phi[lay.phi_off[s]:lay.phi_off[s] + n * lay.ld_phi[s]].view(n, -1)[:, :k] = torch.from_numpy(phi).cuda()
        b.mass[lay.mass_off[s]:lay.mass_off[s] + n] = torch.from_numpy(mass).cuda()
        lay.feat_view(b.feat, s).copy_(f)
        refs.append(phi.T.astype(np.float64) @ (mass[:, None].astype(np.float64) * f.double().numpy()))
    b.project()
    for s, ref in enumerate(refs):
        err = np.linalg.norm(b.a_view(b.A, s).double().cpu().numpy() - ref) / np.linalg.norm(ref)
        assert err <= (2e-5 if feat == "bf16" else 2e-6), (ns[s], ks[s], ds[s], err)


@pytest.mark.parametrize("feat", ["bf16", "fp32"])
@pytest.mark.parametrize("d", [16, 128, 144, 256, 272, 384, 512, 528])
def test_basis_and_feature_edges(d, feat):
    ks = [1, 15, 16, 17, 32, 33, 48, 64, 65, 80, 81, 96, 112, 113, 128, 129, 160, 208, 256, 257]
    _check([300 + 7 * k for k in ks], ks, [d] * len(ks), feat)


@pytest.mark.parametrize("feat", ["bf16", "fp32"])
@pytest.mark.parametrize("ns", [[1], [63, 64, 65], [2100], [40000], [513, 1, 9000, 31]])
def test_partials(ns, feat):
    _check(ns, [20 + 30 * i for i in range(len(ns))], [128] * len(ns), feat)
