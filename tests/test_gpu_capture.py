"""Calls on a stream that the caller is capturing: what the captured graph
computes, and what later calls on the same handle take from its caches."""
import contextlib
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

THREAD_LOCAL, RELAXED = 1, 2


def _cudart():
    for name in ("libcudart.so.13", "libcudart.so", "/usr/local/cuda/lib64/libcudart.so"):
        with contextlib.suppress(OSError):
            return ctypes.CDLL(name)
    pytest.skip("no CUDA runtime library to capture with")


class _Capture:
    """A capture of `stream`; after it, run() launches what was captured (None
    when the capture ended in an error)."""

    def __init__(self, stream, mode=THREAD_LOCAL):
        self.rt, self.s, self.mode = _cudart(), ctypes.c_void_p(stream.cuda_stream), mode
        self.graph = self.exec = None

    def __enter__(self):
        torch.cuda.synchronize()
        assert self.rt.cudaStreamBeginCapture(self.s, self.mode) == 0
        return self

    def __exit__(self, *exc):
        g, x = ctypes.c_void_p(), ctypes.c_void_p()
        if self.rt.cudaStreamEndCapture(self.s, ctypes.byref(g)) == 0 and g.value:
            assert self.rt.cudaGraphInstantiate(ctypes.byref(x), g, ctypes.c_ulonglong(0)) == 0
            self.rt.cudaGraphDestroy(g)
            self.exec = x
        else:
            self.rt.cudaGetLastError()
        return False

    def run(self):
        assert self.rt.cudaGraphLaunch(self.exec, self.s) == 0
        assert self.rt.cudaStreamSynchronize(self.s) == 0

    def close(self):
        if self.exec is not None:
            self.rt.cudaGraphExecDestroy(self.exec)


def _series(n, seed):
    return np.cumsum(np.random.default_rng(seed).standard_normal(n)).astype(np.float32)


class _Call:
    """A device query of one length with outputs of its own."""

    def __init__(self, x, m, seed, r=None):
        rng = np.random.default_rng(seed)
        at = int(rng.integers(0, x.size - m))
        self.q = torch.from_numpy((x[at:at + m] + 0.1 * rng.standard_normal(m)).astype(np.float32)).cuda()
        self.r = m // 10 if r is None else r
        self.out = (torch.zeros(1, dtype=torch.int64, device="cuda"), torch.zeros(1, dtype=torch.float32, device="cuda"))

    def __call__(self, ix, s):
        ix.query(self.q, self.r, out=self.out, stream=s)

    def take(self):
        torch.cuda.synchronize()
        got = int(self.out[0]), float(self.out[1])
        self.out[0].fill_(-1)
        self.out[1].zero_()
        torch.cuda.synchronize()
        return got


@pytest.mark.parametrize("mode", [THREAD_LOCAL, RELAXED])
@pytest.mark.parametrize("options", [dict(), dict(batch_graph=0), dict(exact_envelope=0, batch_graph=0)])
def test_a_length_first_met_under_capture(mode, options):
    """The caches are full and their stream is under capture: the statistics of
    a new length are not computed then, so no later call may take them for
    computed.  Where CUDA lets the capture allocate, the captured search is
    whole."""
    from paper_1812_10302_gb300 import dtws

    x = _series(40_000, 8)
    s = torch.cuda.Stream()
    calls = [_Call(x, m, m) for m in (64, 96, 128, 160, 192, 224, 256, 288, 320, 352)]
    new = _Call(x, 500, 9, r=77)
    with dtws.Index(x, options=options) as ix:
        new(ix, s)
        want = new.take()
    with dtws.Index(x, options=options) as ix:
        for c in calls:
            c(ix, s)
        cap = _Capture(s, mode)
        with cap, contextlib.suppress(dtws.DtwsError):
            new(ix, s)
        new(ix, s)  # (before any run of the captured graph)
        assert new.take() == want
        if cap.exec is not None and options:  # (a repeated search is a graph of its own: refused unless it ran last)
            cap.run()
            assert new.take() == want
            calls[0](ix, s)
            cap.run()
            assert new.take() == want
        cap.close()
        assert ix.sync_status() == dtws.DTWS_OK


@pytest.mark.parametrize("before", [1, 2, 3])
@pytest.mark.parametrize("options", [dict(), dict(batch_graph=0), dict(exclusion_zone=4)])
def test_a_captured_search_outlives_the_caches_slots(before, options):
    """A search that ran once, twice (captured by the handle) or three times
    (replayed by it) is taken by the caller's capture; the captured graph gives
    the same answer after more lengths, bands and larger arrays than the
    handle's caches and its stage hold."""
    from paper_1812_10302_gb300 import dtws

    x = _series(40_000, 18)
    s = torch.cuda.Stream()
    one = _Call(x, 128, 3)
    with dtws.Index(x, options=options) as ix:
        for _ in range(before):
            one(ix, s)
        want = one.take()
        cap = _Capture(s)
        with cap:
            one(ix, s)
        cap.run()
        assert one.take() == want
        one(ix, s)
        assert one.take() == want
        for rep in range(2):
            for m in (64, 96, 160, 192, 224, 256, 288, 320, 352, 384, 6000):
                ix.query(x[100:100 + m], m // 7, stream=s)
            cap.run()
            assert one.take() == want
        one(ix, s)
        assert one.take() == want
        cap.close()
        assert ix.sync_status() == dtws.DTWS_OK


def test_a_captured_learned_search_outlives_its_slots():
    """The embeddings that a captured search reads stay too."""
    from oracle import encoder as enc
    from paper_1812_10302_gb300 import dtws, synth

    x = synth.walk_with_bursts(300_000, 71, 72, 73)
    s = torch.cuda.Stream()
    one = _Call(x, 128, 4)
    with dtws.Index(x) as ix:
        ix.set_encoder(enc.init_params(3))
        ix.set_options(ordering=dtws.DTWS_ORDER_LEARNED)
        one(ix, s)
        want = one.take()
        cap = _Capture(s)
        with cap:
            one(ix, s)
        for m in (64, 192, 256, 320, 64, 192):
            ix.query(x[100:100 + m], m // 7, stream=s)
        cap.run()
        assert one.take() == want
        ix.set_encoder(enc.init_params(4))
        for m in (64, 192, 256, 320, 128):
            ix.query(x[100:100 + m], m // 7, stream=s)
        cap.run()
        assert one.take() == want
        cap.close()
        assert ix.sync_status() == dtws.DTWS_OK


def test_other_searches_are_refused_under_capture():
    """Under capture a handle that keeps graphs takes no search but the last one
    and the one whose graph it keeps, and is as it was afterwards."""
    from paper_1812_10302_gb300 import dtws

    x = _series(30_000, 28)
    s = torch.cuda.Stream()
    a, b, c = (_Call(x, m, m) for m in (100, 200, 300))
    with dtws.Index(x) as ix:
        want = {}
        for call in (a, a, c, b):  # a's graph is kept, b ran last
            call(ix, s)
            want[call] = call.take()
        for call, taken in ((a, True), (b, True), (c, False)):
            cap = _Capture(s)
            with cap:
                if taken:
                    call(ix, s)
                else:
                    with pytest.raises(dtws.DtwsError):
                        call(ix, s)
            if taken:
                cap.run()
                assert call.take() == want[call]
            cap.close()
        for call in (a, b, c, c, a):
            call(ix, s)
            assert call.take() == want[call]
