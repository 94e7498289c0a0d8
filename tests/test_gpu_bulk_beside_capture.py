"""A bulk call on one stream while another stream, of the same or another thread, is
being captured: it takes scratch memory of its own, and neither the call nor the
capture may fail for it."""
import threading

import pytest
import torch

from paper_1908_05936_gb300 import _lib as L
from paper_1908_05936_gb300.table import Table
from test_gpu_bulk import keys_of, vals_of

pytestmark = pytest.mark.gpu

N = 2 * (800 << 20) // 128


@pytest.mark.parametrize("mode", ("global", "thread_local", "relaxed"))
def test_capture_on_another_stream(mode):
    t = Table(L.MAP_U64_U64, (800 << 20) // 16, bucket_bytes=64)
    try:
        k = keys_of(torch.arange(N, device="cuda"), L.MAP_U64_U64)
        v = vals_of(k, L.MAP_U64_U64)
        st, f, w = torch.ones(N, dtype=torch.uint8, device="cuda"), torch.zeros(N, dtype=torch.uint8, device="cuda"), torch.empty_like(k)
        x = torch.zeros(8, device="cuda")
        side, other = torch.cuda.Stream(), torch.cuda.Stream()
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=side, capture_error_mode=mode):
            x += 1
            t.insert(k, v, status=st, stream=other)
            t.find(k, found=f, vals_out=w, stream=other)
            x += 1
        torch.cuda.synchronize()
        g.replay()
        torch.cuda.synchronize()
        assert float(x.sum()) == 16.0
        assert not bool(st.any()) and bool(f.all()) and torch.equal(w, v)
    finally:
        t.close()


def test_capture_in_another_thread():
    t = Table(L.MAP_U64_U64, (800 << 20) // 16, bucket_bytes=64)
    try:
        k = keys_of(torch.arange(N, device="cuda"), L.MAP_U64_U64)
        f = torch.zeros(N, dtype=torch.uint8, device="cuda")
        x = torch.zeros(8, device="cuda")
        other = torch.cuda.Stream()
        t.insert(k, vals_of(k, L.MAP_U64_U64), status=False)
        torch.cuda.synchronize()
        started, called, failed = threading.Event(), threading.Event(), []
        g = torch.cuda.CUDAGraph()

        def capture():
            try:
                with torch.cuda.graph(g, stream=torch.cuda.Stream(), capture_error_mode="global"):
                    x.add_(1)
                    started.set()
                    called.wait(60)
            except Exception as e:                              # noqa: BLE001 (handed to the test's thread)
                failed.append(e)
                started.set()

        th = threading.Thread(target=capture)
        th.start()
        assert started.wait(60)
        t.find(k, found=f, vals_out=False, stream=other)
        called.set()
        th.join()
        torch.cuda.synchronize()
        assert not failed, failed
        g.replay()
        torch.cuda.synchronize()
        assert float(x.sum()) == 8.0 and bool(f.all())
    finally:
        t.close()
