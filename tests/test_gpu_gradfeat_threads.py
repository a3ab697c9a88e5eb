"""Gradient features of different widths from two threads at once, each on its own stream: neither takes
from the other the shared memory that its kernel launches with."""
import ctypes
import threading

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_two_widths_from_two_threads():
    from paper_2604_10377_gb300 import _lib, api
    n, per_row = 200, 5
    rng = np.random.default_rng(0)
    ptr = torch.from_numpy((per_row * np.arange(n + 1)).astype(np.int64)).cuda()
    col = torch.from_numpy(rng.integers(0, n, n * per_row).astype(np.int32)).cuda()
    vals = torch.from_numpy(rng.standard_normal((n * per_row, 2)).astype(np.float32)).cuda()
    start, failed = threading.Barrier(2, timeout=60), []

    def work(dim):
        try:
            draw = np.random.default_rng(dim)
            x, ar, ai = (torch.from_numpy(draw.standard_normal(s).astype(np.float32)).cuda()
                         for s in ((n, dim), (dim, dim), (dim, dim)))
            st = torch.cuda.Stream()
            st.wait_stream(torch.cuda.default_stream())
            with torch.cuda.stream(st):
                want = api.gradient_features(ptr, col, vals, x, ar, ai)[0]
                out, status = torch.zeros_like(want), torch.zeros(1, dtype=torch.int32, device="cuda")
                ws = torch.empty(1 << 20, dtype=torch.uint8, device="cuda")
            p = [ctypes.c_void_p(t.data_ptr()) for t in (ptr, col, vals, x, ar, ai, out, status, ws)]
            call = _lib.lib().fmap_gradient_features
            args = (n, p[0], p[1], p[2], n * per_row, n, p[3], dim, dim, p[4], p[5], 0, p[6], dim, 0, p[7], p[8],
                    ws.numel(), ctypes.c_void_p(st.cuda_stream))
            start.wait()
            codes = {call(*args) for _ in range(4000)}     # (nothing but the calls: they have to overlap)
            st.synchronize()
            assert codes == {0} and int(status) == 0 and torch.equal(out, want)
        except Exception as e:          # reported by the main thread
            failed.append((dim, e))

    threads = [threading.Thread(target=work, args=(dim,)) for dim in (16, 128)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed
