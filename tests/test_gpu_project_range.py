"""FP32 projections of operands near the largest FP32 number: their heads must not round to infinity. Products
and sums stay far inside the range, so the tolerances are those of ordinary inputs (forward 2e-6, backward
1e-5, against FP64); infinities and NaN stay non-finite in the rows they reach and nowhere else."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

N, K, D = 700, 40, 48
BIG = [3.3970e38, 3.4015e38]


def _batch():
    from paper_2604_10377_gb300 import api
    lay = api.BatchLayout([N], [K], [D], "fp32")
    b = api.FmapBatch(lay, [(0, 0, 1e-2)], precision="fp32")
    return lay, b


def _big(rng, shape, value):
    x = (value * rng.uniform(0.25, 1.0, shape)).astype(np.float32)
    x[rng.random(shape) < 0.5] = np.float32(value)
    x[rng.random(shape) < 0.5] *= -1
    return x


def _run(phi, mass, feat, da):
    lay, b = _batch()
    b.phi.view(-1)[:N * lay.ld_phi[0]].view(N, -1)[:, :K] = torch.from_numpy(phi).cuda()
    b.mass[:N] = torch.from_numpy(mass).cuda()
    lay.feat_view(b.feat, 0).copy_(torch.from_numpy(feat))
    a = b.a_view(b.project(), 0).cpu().numpy()
    b.a_view(b.dA, 0).copy_(torch.from_numpy(da))
    b.project_backward()
    return a, lay.feat_view(b.dfeat, 0).cpu().numpy()


def _rel(x, ref):
    return np.linalg.norm(x.astype(np.float64) - ref) / np.linalg.norm(ref)


@pytest.mark.parametrize("value", BIG)
@pytest.mark.parametrize("which", ["feat", "phi", "da"])
def test_operands_near_the_largest_number(which, value):
    rng = np.random.default_rng(len(which))
    tiny = 1e-20
    phi, feat, da = (rng.standard_normal(s).astype(np.float32) for s in ((N, K), (N, D), (K, D)))
    mass = np.ones(N, np.float32)
    if which == "phi":
        phi, feat, da = _big(rng, (N, K), value), feat * np.float32(tiny), da * np.float32(tiny)
    elif which == "feat":
        feat, phi = _big(rng, (N, D), value), phi * np.float32(tiny)
    else:
        da, phi = _big(rng, (K, D), value), phi * np.float32(tiny)
    a, df = _run(phi, mass, feat, da)
    assert _rel(a, phi.T.astype(np.float64) @ feat.astype(np.float64)) <= 2e-6
    assert _rel(df, phi.astype(np.float64) @ da.astype(np.float64)) <= 1e-5


@pytest.mark.parametrize("value", [np.inf, np.nan])
def test_non_finite_features_stay_in_their_columns(value):
    rng = np.random.default_rng(5)
    phi, feat, da = (rng.standard_normal(s).astype(np.float32) for s in ((N, K), (N, D), (K, D)))
    feat[123, 17] = value
    a, _ = _run(phi, np.ones(N, np.float32), feat, da)
    assert not np.isfinite(a[:, 17]).any()
    assert np.isfinite(np.delete(a, 17, 1)).all()
