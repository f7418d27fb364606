"""The walk from both ends (seeds, survivors and the FP32 pre-score on one warp
per window) against the FP64 oracle, at the edges of its shapes (two to
sixteen cells a lane: 32 K >= r + 1, K = 1, 2, 3, 4, 6, 8), both parities of m + r
(where the ends meet), queries hardly longer than the band, and candidates so
close together that few can be abandoned."""
import numpy as np
import pytest

import oracle
from paper_1812_10302_gb300 import dtws, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,r", [(17, 16), (18, 16), (33, 31), (34, 32), (64, 63), (65, 63), (66, 64), (97, 95), (100, 96),
                                 (128, 127), (129, 127), (140, 128), (193, 191), (200, 192), (256, 255), (400, 255),
                                 (333, 40), (334, 41), (1024, 102)])
@pytest.mark.parametrize("exact_envelope", [0, 1])
def test_answers_at_shape_edges(m, r, exact_envelope):
    x = synth.random_walk(6_000, m + r)
    x[1000:5000] = np.sin(np.arange(4000) / 30.0) * 5 + 0.3 * x[1000:5000]  # many near ties
    q, _ = synth.noisy_copy(x, m, m, r, noise=0.2)
    with dtws.Index(x, options=dict(exact_envelope=exact_envelope)) as ix:
        idx, dist = ix.query(q, r, 5)
        assert ix.sync_status() == dtws.DTWS_OK
        bi, bd = ix.query_batch([q, q[: m - 1]], [r, min(r, m - 2)], 5)
    oi, od = oracle.search_cascade(x, q, r, 5)
    np.testing.assert_array_equal(idx, oi)
    np.testing.assert_allclose(dist, od, rtol=1e-6)
    np.testing.assert_array_equal(bi[0], oi)
    np.testing.assert_allclose(bd[0], od, rtol=1e-6)


@pytest.mark.parametrize("m,r", [(513, 512), (620, 512), (609, 608), (611, 609), (700, 610), (1097, 1096), (1100, 1097),
                                 (1099, 1098), (1585, 1584), (1590, 1585), (2048, 2047), (2100, 2047), (1024, 921)])
def test_overlapping_warps(m, r):
    """The walk over four warps at the widest band of each cell count (122 K >
    r, K = 5, 9, 13, 17) and the first past it, both parities, with and without
    abandoning; the pre-score's shapes beside it."""
    x = synth.random_walk(3 * m, m + r)
    q, o = synth.noisy_copy(x, m, m, r, noise=0.2)
    offs = np.array([o, 0, x.size - m, m // 2, m + 1])
    with dtws.Index(x) as ix:
        got = ix.dtw_at(q, r, offs)
        idx, dist = ix.query(q, r, 2)
        one, d1 = ix.query(q, r, 1)
        assert ix.sync_status() == dtws.DTWS_OK
    np.testing.assert_allclose(got, oracle.dtw_at(x, q, r, offs), rtol=1e-4, atol=1e-6 * m)
    oi, od = oracle.search_cascade(x, q, r, 2)
    np.testing.assert_array_equal(idx, oi)
    np.testing.assert_allclose(dist, od, rtol=1e-6)
    assert one[0] == oi[0]
    np.testing.assert_allclose(d1[0], od[0], rtol=1e-6)


@pytest.mark.parametrize("m,r", [(64, 5), (64, 20), (128, 60), (200, 142), (400, 300), (600, 560)])
@pytest.mark.parametrize("k", [2, 5])
def test_no_window_is_scored_twice(m, r, k):
    """With no more windows than the exact seeds reach, every window is scored
    once: the best Euclidean seed is one of them, and a second score, rounded
    in another order, could put it into the list of results twice."""
    x = synth.random_walk(m + k, m + r)
    q, _ = synth.noisy_copy(x, m, m, r, noise=0.3)
    with dtws.Index(x) as ix:
        idx, dist = ix.query(q, r, k)
        assert ix.sync_status() == dtws.DTWS_OK
        assert ix.last_stats()["dtw_started"] <= k + 1
    oi, od = oracle.search_cascade(x, q, r, k)
    np.testing.assert_array_equal(idx, oi)
    np.testing.assert_allclose(dist, od, rtol=1e-6)
