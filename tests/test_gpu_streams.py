"""One handle's calls on several streams, none of which the caller waits for:
every answer is the one a handle of its own gives."""
import ctypes
import threading

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1812_10302_gb300 import dtws, synth  # noqa: E402

pytestmark = pytest.mark.gpu

N = 3_000_000
PER_THREAD = 2  # the handle of every thread's own default stream


@pytest.fixture(scope="module")
def series():
    return torch.from_numpy(synth.walk_with_bursts(N, 91, 92, 93)).cuda()


class _Search:
    def __init__(self, x, m, r, k, seed):
        g = torch.Generator(device="cuda").manual_seed(seed)
        at = (seed * 7919 + m) % (x.numel() - m)
        self.q = x[at:at + m] + 0.2 * torch.randn(m, generator=g, device="cuda")
        self.r, self.k = r, k
        self.out = (torch.zeros(k, dtype=torch.int64, device="cuda"), torch.zeros(k, dtype=torch.float32, device="cuda"))
        with dtws.Index(x) as ix:
            self.want = ix.query(self.q, r, k)
        self.want = [np.asarray(torch.as_tensor(w).cpu()) for w in self.want]

    def __call__(self, ix, stream):
        ix.query(self.q, self.r, self.k, out=self.out, stream=stream)

    def check(self):
        np.testing.assert_array_equal(self.out[0].cpu().numpy(), self.want[0])
        np.testing.assert_array_equal(self.out[1].cpu().numpy(), self.want[1])
        self.out[0].fill_(-1)


def _searches(x):
    shapes = [(300, 280, 1), (1024, 921, 1), (512, 51, 10), (128, 6, 1), (600, 520, 4), (900, 90, 1), (64, 60, 8)]
    return [_Search(x, m, r, k, 10 + i) for i, (m, r, k) in enumerate(shapes)]


@pytest.mark.parametrize("batch_graph", [0, 1])
def test_searches_on_alternating_streams(series, batch_graph):
    """Searches and distances at offsets in turn on three streams, queued
    without a wait, each search three times."""
    todo = _searches(series)
    offs = torch.arange(0, N - 2000, 5003, device="cuda")
    streams = [torch.cuda.Stream(), torch.cuda.default_stream(), torch.cuda.Stream()]
    with dtws.Index(series, options=dict(batch_graph=batch_graph)) as ix:
        far = ix.dtw_at(todo[0].q, 280, offs)
        got = torch.zeros(offs.numel(), device="cuda")
        torch.cuda.synchronize()
        t = 0
        for rep in range(3):
            for a in todo:
                for _ in range(3):
                    a(ix, streams[t % 3])
                    t += 1
                assert dtws.load().dtws_dtw_at(ix.h, todo[0].q.data_ptr(), 300, 280, offs.data_ptr(), offs.numel(),
                                               got.data_ptr(), streams[t % 3].cuda_stream) == dtws.DTWS_OK
            torch.cuda.synchronize()
            for a in todo:
                a.check()
            np.testing.assert_array_equal(got.cpu().numpy(), far)
        assert ix.sync_status() == dtws.DTWS_OK


_room = []


def _evict(ix, stream):
    """Statistics and envelopes of more lengths and bands than a handle keeps, on `stream`."""
    lib, s = dtws.load(), dtws._stream_ptr(stream)
    while len(_room) < 3:
        _room.append(torch.empty(N, device="cuda"))
    p = [t.data_ptr() for t in _room]
    for m in range(40, 52):
        assert lib.dtws_window_stats(ix.h, m, *p, s) == dtws.DTWS_OK
        assert lib.dtws_series_envelope(ix.h, m, p[0], p[1], s) == dtws.DTWS_OK


def test_slots_are_rewritten_after_their_readers(series):
    """Searches queued on one stream, then every slot of the caches rewritten on
    another."""
    todo = _searches(series)[2:5]
    a, b = torch.cuda.Stream(), torch.cuda.Stream()
    with dtws.Index(series) as ix:
        _evict(ix, b)
        for s in todo:
            torch.cuda.synchronize()
            for _ in range(20):
                s(ix, a)
            _evict(ix, b)
            torch.cuda.synchronize()
            s.check()


def test_per_thread_default_streams(series):
    """Two threads, one after the other, each on its own default stream: one
    handle value, two streams."""
    todo = _searches(series)[2:5]
    with dtws.Index(series) as ix:
        _evict(ix, PER_THREAD)
        for s in todo:
            torch.cuda.synchronize()

            def search():
                for _ in range(20):
                    s(ix, PER_THREAD)

            for work in (search, lambda: _evict(ix, PER_THREAD), search, lambda: todo[0](ix, PER_THREAD)):
                t = threading.Thread(target=work)
                t.start()
                t.join()
            torch.cuda.synchronize()
            s.check()


def test_a_stream_that_is_gone(series):
    """Searches queued on a stream that is destroyed before they have run; the
    next stream may get its handle."""
    try:
        rt = ctypes.CDLL("libcudart.so.13")
    except OSError:
        rt = ctypes.CDLL("/usr/local/cuda/lib64/libcudart.so")
    todo = _searches(series)[2:5]
    with dtws.Index(series) as ix:
        torch.cuda.synchronize()
        for rep in range(4):
            for s in todo:
                h = ctypes.c_void_p()
                assert rt.cudaStreamCreateWithFlags(ctypes.byref(h), 1) == 0
                for _ in range(6):
                    s(ix, h.value)
                assert rt.cudaStreamDestroy(h) == 0
            torch.cuda.synchronize()
            for s in todo:
                s.check()
