"""The query preparation's envelope and ordered terms and the lower-bound
scan's forms (one window at a time, several lanes at a time, whole rows) at the
sizes where they change: queries shorter and longer than the 128 terms, bands
from 0 to the whole query, thresholds from tight to so loose that most windows
pass, against the FP64 oracle."""
import numpy as np
import pytest

import oracle
from paper_1812_10302_gb300 import dtws, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def series():
    return synth.random_walk(30_000, 25)


@pytest.mark.parametrize("m,r", [(2, 0), (2, 1), (3, 1), (3, 2), (5, 4), (33, 16), (66, 1), (129, 3), (130, 129),
                                 (131, 64), (257, 31), (1024, 921), (2048, 2047), (8192, 0), (8192, 4000)])
def test_query_envelope_bound(series, m, r):
    """Eq. 8 in full: FP32 sums of at most m squared terms, each rounded to
    2^-22 relative."""
    q, _ = synth.noisy_copy(series, m, m + r, m, noise=0.3)
    offs = np.random.default_rng(m + r).integers(0, series.size - m + 1, 200)
    with dtws.Index(series) as ix:
        _, kq, _ = ix.lower_bounds_at(q, r, offs)
    _, okq, _, _ = oracle.lbs_at(series, q, r, offs)
    np.testing.assert_allclose(kq, okq, rtol=1e-4, atol=1e-5 * m)


@pytest.mark.parametrize("m,r", [(2, 1), (3, 0), (4, 3), (8, 2), (34, 3), (65, 6), (66, 5), (67, 60), (129, 12), (130, 13),
                                 (131, 2), (500, 50)])
@pytest.mark.parametrize("k,proposals", [(1, 16), (1, 0), (64, 16), (7, 0)])
def test_search_tight_and_loose(series, m, r, k, proposals):
    """proposals = 0 leaves only random windows to start from, so that nearly
    every window passes LB_KimFL."""
    q, _ = synth.noisy_copy(series, m, 3 * m + r, m + 1, noise=0.2)
    with dtws.Index(series, options=dict(seed_proposals=proposals)) as ix:
        idx, dist = ix.query(q, r, k)
        assert ix.sync_status() in ((dtws.DTWS_OK, dtws.DTWS_EOVERFLOW) if m < 8 else (dtws.DTWS_OK,))
    oi, od = oracle.search_cascade(series, q, r, k)
    if m >= 8:  # (below, many windows tie within rounding)
        np.testing.assert_array_equal(idx, oi)
    np.testing.assert_allclose(dist, od, rtol=1e-4, atol=1e-6 * m)


@pytest.mark.parametrize("n,m", [(1024, 600), (4096 + 511, 512), (5000, 16), (200_003, 128)])
def test_seeds_from_few_and_ragged_tiles(n, m):
    """One to a few proxy tiles, scan warps without a window, a ragged last
    tile: the answer is the planted window wherever it lies."""
    x = synth.random_walk(n, n)
    rng = np.random.default_rng(m)
    for o in (0, n - m, (n - m) // 2, (n - m) // 3):
        q = (x[o:o + m].astype(np.float64) + rng.normal(0, 0.02, m)).astype(np.float32)
        with dtws.Index(x) as ix:
            idx, dist = ix.query(q, max(1, m // 20), 1)
            assert ix.sync_status() == dtws.DTWS_OK
            bsf = ix.last_stats()["seed_bsf"]
        d = oracle.dtw_at(x, q, max(1, m // 20), [o])[0]
        assert idx[0] == o
        np.testing.assert_allclose(dist, d, rtol=1e-4, atol=1e-6 * m)
        assert bsf >= d * (1 - 1e-3) - 1e-6 * m  # a Euclidean distance: an upper bound


@pytest.mark.parametrize("m,r", [(64, 40), (65, 33), (65, 64), (66, 50), (97, 96), (300, 31), (300, 35), (513, 512),
                                 (600, 520), (1025, 1000), (1100, 1099)])
@pytest.mark.parametrize("k", [1, 6])
def test_corner_bound_keeps_every_answer(series, m, r, k):
    """Bands from the narrowest that one warp walks (32 lanes) to the whole
    query, query lengths around twice the corner, with and without a tight
    first bound."""
    x = series[:9000]
    q, _ = synth.noisy_copy(x, m, 5 * m + r, m + 3, noise=0.4)
    oi, od = oracle.search_cascade(x, q, r, k)
    for proposals in (16, 0):
        with dtws.Index(x, options=dict(seed_proposals=proposals)) as ix:
            idx, dist = ix.query(q, r, k)
            assert ix.sync_status() == dtws.DTWS_OK
        np.testing.assert_array_equal(idx, oi)
        np.testing.assert_allclose(dist, od, rtol=1e-4, atol=1e-6 * m)
