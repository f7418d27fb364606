"""The wide exclusion zone's bucket lists: many windows offered at once, every
length of list, against the FP64 oracle's greedy selection."""
import numpy as np
import pytest

import oracle
from paper_1812_10302_gb300 import dtws, synth

pytestmark = pytest.mark.gpu


def test_offers_do_not_queue_for_long():
    """A loose bound: most windows that are walked are offered.  No offer waits
    half a second for its list's lock (all of them together took 1.9 s, one
    after another, when every waiter asked again every 64 ns)."""
    n, m, k, z = 1_000_000, 128, 64, 64
    x = synth.random_walk(n, n + m)
    q, _ = synth.noisy_copy(x, m, m, k, noise=0.2)
    with dtws.Index(x, options=dict(exclusion_zone=z, wait_limit_ns=500_000_000)) as ix:
        idx, dist = ix.query(q, m // 10, k)
        assert ix.sync_status() == dtws.DTWS_OK
    assert np.all(np.diff(np.sort(idx)) > z)
    np.testing.assert_allclose(dist, oracle.dtw_at(x, q, m // 10, idx), rtol=1e-4, atol=1e-6 * m)


@pytest.mark.parametrize("k,z", [(1, 40), (2, 40), (7, 33), (8, 33), (9, 64), (16, 20), (40, 12), (63, 16), (64, 16), (64, 300)])
@pytest.mark.parametrize("kind", ["walk", "ties"])
def test_lists_of_every_length(k, z, kind):
    """List lengths around the eight entries read at a time and the longest;
    "ties": runs of windows within rounding of each other, many to a bucket."""
    n, m, r = 12_000, 64, 6
    x = synth.random_walk(n, 640 + k)
    if kind == "ties":
        x = (np.sin(np.arange(n) / 9.0) * 3 + 0.02 * x).astype(np.float32)
    q, _ = synth.noisy_copy(x, m, 641, 642 + k, noise=0.2)
    d = oracle.dtw_at(x, q, r, np.arange(n - m + 1))
    oi, od = oracle.exclusion_topk(d, k, z)
    with dtws.Index(x, options=dict(exclusion_zone=z)) as ix:
        for _ in range(3):
            idx, dist = ix.query(q, r, k)
            if oi.size < k:  # no k windows far enough apart, so no bound: more candidates than the re-score list's 8192
                assert ix.sync_status() == dtws.DTWS_EOVERFLOW
                return
            assert ix.sync_status() == dtws.DTWS_OK
            np.testing.assert_array_equal(idx, oi)
            np.testing.assert_allclose(dist, od, rtol=1e-4, atol=1e-6 * m)


@pytest.mark.parametrize("n,m,k,z", [(200_000, 128, 20, 200), (30_000, 64, 6, 100)])
def test_a_short_series_has_a_first_bound(n, m, k, z):
    """The seeds of a short series hold k windows far enough apart, so that the
    scan has a bound: without one every window passes it."""
    x = synth.random_walk(n, n + m)
    q, _ = synth.noisy_copy(x, m, m, k, noise=0.2)
    with dtws.Index(x, options=dict(exclusion_zone=z)) as ix:
        idx, dist = ix.query(q, m // 10, k)
        assert ix.sync_status() == dtws.DTWS_OK
        assert ix.last_stats()["pass_keogh_q"] < 0.9 * (n - m + 1)
    assert np.all(np.diff(np.sort(idx)) > z)
    np.testing.assert_allclose(dist, oracle.dtw_at(x, q, m // 10, idx), rtol=1e-4, atol=1e-6 * m)
