"""Two batches of different sizes alive at once: creating the smaller one must not take from the larger
one's kernels the shared memory that they launch with."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _batch(n, k, d, feat):
    from paper_2604_10377_gb300 import api
    lay = api.BatchLayout([n, n], [k, k], [d, d], feat)
    b = api.FmapBatch(lay, [(0, 1, 1e-2)], precision=feat)
    g = torch.Generator(device="cuda").manual_seed(k)
    b.phi.normal_(generator=g)
    b.mass.fill_(1.0 / n)
    b.feat.normal_(generator=g)
    b.dA.normal_(generator=g)
    return b


@pytest.mark.parametrize("feat", ["fp32", "bf16"])
@pytest.mark.parametrize("k,d", [(300, 512), (200, 512), (100, 512), (40, 256)])
def test_smaller_batch_leaves_the_larger_one_running(k, d, feat):
    large = _batch(1000, k, d, feat)
    a = large.project().clone()
    large.project_backward()
    df = large.dfeat.clone()
    small = _batch(300, 8, 16, feat)
    small.project()
    small.project_backward()
    large.A.zero_()
    large.dfeat.zero_()
    assert torch.equal(large.project(), a)
    large.project_backward()
    assert torch.equal(large.dfeat, df)
