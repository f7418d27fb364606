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
