"""The handle's caches when their slots are reused and its streams differ."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


def _fresh(x, q, r):
    from paper_1812_10302_gb300 import dtws

    with dtws.Index(x) as ix:
        i, d = ix.query(q, r=r)
        return int(i[0]), float(d[0])


@pytest.mark.parametrize("streams", [1, 2])
def test_reused_slots_hold_the_new_lengths_statistics(streams):
    """Twelve lengths and bands over fewer slots, longest and shortest in turn
    (a slot's tail then holds another length's values), each query repeated
    three times in a row (launched, captured, replayed)."""
    from paper_1812_10302_gb300 import dtws

    rng = np.random.default_rng(5)
    x = np.cumsum(rng.standard_normal(20001)).astype(np.float32)
    lengths = [2048, 2, 1500, 17, 1024, 33, 700, 64, 513, 129, 300, 255]
    ss = [torch.cuda.Stream() for _ in range(streams)]
    with dtws.Index(x) as ix:
        for rep in range(2):
            for t, m in enumerate(lengths):
                q = (x[5000 : 5000 + m] + 0.1 * rng.standard_normal(m)).astype(np.float32)
                r = min(m - 1, 1 + 7 * t)
                want = _fresh(x, q, r)
                s = ss[(t + rep) % streams]
                for _ in range(3):
                    i, d = ix.query(q, r=r, stream=s)
                    assert (int(i[0]), float(d[0])) == want, (m, r)


def test_query_seen_once_is_taken_under_capture():
    """A device query that has run once is accepted by a stream under capture
    and gives the same answer on replay."""
    from paper_1812_10302_gb300 import dtws

    rng = np.random.default_rng(6)
    x = np.cumsum(rng.standard_normal(30000)).astype(np.float32)
    q = torch.from_numpy((x[7000:7128] + 0.05 * rng.standard_normal(128)).astype(np.float32)).cuda()
    oi = torch.zeros(1, dtype=torch.int64, device="cuda")
    od = torch.zeros(1, dtype=torch.float32, device="cuda")
    with dtws.Index(torch.from_numpy(x).cuda()) as ix:
        s = torch.cuda.Stream()
        with torch.cuda.stream(s):
            ix.query(q, r=12, out=(oi, od), stream=s)
        s.synchronize()
        want = (int(oi), float(od))
        oi.zero_(), od.zero_()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            ix.query(q, r=12, out=(oi, od), stream=s)
        g.replay()
        torch.cuda.synchronize()
        assert (int(oi), float(od)) == want


def test_a_kept_graph_does_not_outlive_its_embeddings():
    """Learned ordering, two slots of embeddings: a query is captured, another
    length takes its slot and a third one brings the first length back to the
    same place of the cache, at other addresses.  The plain ordering's answers
    every time."""
    from oracle import encoder as enc
    from paper_1812_10302_gb300 import dtws, synth

    x = synth.walk_with_bursts(400_000, 61, 62, 63)
    qs = {m: synth.noisy_copy(x, m, 64 + m, 65 + m, noise=0.2)[0] for m in (64, 128, 256)}
    with dtws.Index(x) as ix:
        want = {m: ix.query(q, m // 10) for m, q in qs.items()}
    with dtws.Index(x) as ix:
        ix.set_encoder(enc.init_params(3))
        ix.set_options(ordering=dtws.DTWS_ORDER_LEARNED)
        for m in (64, 128, 128, 256, 64, 128, 128, 128, 256, 256, 64, 128, 256):
            i, d = ix.query(qs[m], m // 10)
            assert ix.sync_status() == dtws.DTWS_OK
            np.testing.assert_array_equal(i, want[m][0])
            np.testing.assert_array_equal(d, want[m][1])
