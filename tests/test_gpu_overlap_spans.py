"""Overlap counts over equal spans of the flat vertex range: segments shorter and longer than a
warp's span, empty segments at either end and in between, ranges that start past zero, and score
and label arrays whose 4-vertex alignments agree or not. The counts are integers: exact."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _lengths(kind, rng):
    if kind == "one_vertex":
        return [1]
    if kind == "short":
        return list(rng.integers(0, 7, 3000))
    if kind == "empty_ends":
        return [0, 0, 5, 0, 0, 1023, 1024, 1025, 0]
    if kind == "mixed":
        return [3, 70001, 0, 1, 4095, 4096, 4097, 31, 1200003, 2]
    return list(rng.integers(900, 30000, 700))


@pytest.mark.parametrize("kind", ["one_vertex", "short", "empty_ends", "mixed", "many"])
@pytest.mark.parametrize("lead,shift_s,shift_l", [(0, 0, 0), (5, 1, 1), (3, 2, 0), (0, 3, 1)])
def test_counts_are_exact(kind, lead, shift_s, shift_l):
    from paper_2604_10377_gb300 import api
    rng = np.random.default_rng(len(kind) + 10 * lead + shift_s)
    off = lead + np.concatenate([[0], np.cumsum(_lengths(kind, rng))]).astype(np.int64)
    n = int(off[-1]) + 9
    scores = rng.random(n, dtype=np.float32)
    scores[rng.random(n) < 0.05] = 0.5          # equal to the threshold: not above it
    scores[rng.random(n) < 0.02] = np.nan
    labels = rng.choice(np.array([0, 0, 1, 7, 255], np.uint8), n)
    s_dev = torch.zeros(n + shift_s, device="cuda")[shift_s:]
    l_dev = torch.zeros(n + shift_l, dtype=torch.uint8, device="cuda")[shift_l:]
    s_dev.copy_(torch.from_numpy(scores))
    l_dev.copy_(torch.from_numpy(labels))
    counts, _ = api.overlap_metrics(s_dev, l_dev, off, 0.5)
    with np.errstate(invalid="ignore"):
        pred = scores > np.float32(0.5)
    lab = labels != 0
    want = []
    for m in (pred & lab, pred & ~lab, ~pred & lab, ~pred & ~lab):
        cs = np.concatenate([[0], np.cumsum(m)])
        want.append(cs[off[1:]] - cs[off[:-1]])
    assert np.array_equal(counts.cpu().numpy(), np.stack(want, 1))
