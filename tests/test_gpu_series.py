"""The per-series passes (prefix sums, the one-pass kernel, the block envelope)
at series lengths around their blocks (8192 samples) and tiles, against the
FP64 oracle."""
import numpy as np
import pytest

import oracle
from paper_1812_10302_gb300 import dtws, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [2, 17, 515, 8191, 8192, 8193, 16385, 24576])
@pytest.mark.parametrize("scale", [1.0, 2.0 ** -20, 1e6])
def test_statistics_at_block_edges(n, scale):
    """Every window's mean within 1e-7 sigma and 1/sigma within 2^-22 of the
    two-pass FP64 values, whatever the series' units."""
    x = (synth.random_walk(n, 40 + n).astype(np.float64) * scale).astype(np.float32)
    with dtws.Index(x) as ix:
        for m in sorted({2, min(64, n), min(1000, n), min(8192, n)}):
            mh, ml, inv = ix.window_stats(m)
            mu, sg = oracle.window_stats(x, m, "twopass")
            got = mh.astype(np.float64) + ml.astype(np.float64)
            nz = sg > 0.0
            np.testing.assert_array_equal(inv == 0.0, ~nz)
            assert np.all(np.abs(got[nz] - mu[nz]) <= 1e-7 * sg[nz] + 1e-12 * np.abs(mu[nz]))
            # (1/sigma itself must lie in FP32's range for its relative error to mean anything)
            rel = np.abs(inv[nz].astype(np.float64) * sg[nz] - 1.0)
            assert rel.size == 0 or rel.max() <= 2.0 ** -22


@pytest.mark.parametrize("n", [600, 8192, 16400, 33001])
def test_search_with_the_block_envelope_at_block_edges(n):
    """The sparse table of the block envelope bounds the true envelope at every
    level: the answer with it alone equals the oracle's."""
    x = synth.random_walk(n, 60 + n)
    for m, r in ((64, 3), (256, 200)):
        q, _ = synth.noisy_copy(x, m, n + m, n + r, noise=0.3)
        with dtws.Index(x, options=dict(exact_envelope=0)) as ix:
            idx, dist = ix.query(q, r, 3)
            assert ix.sync_status() == dtws.DTWS_OK
        oi, od = oracle.search_cascade(x, q, r, 3)
        np.testing.assert_array_equal(idx, oi)
        np.testing.assert_allclose(dist, od, rtol=1e-4, atol=1e-6 * m)


@pytest.mark.parametrize("n,at", [(5, 4), (8192, 8191), (8193, 8192), (20_000, 0)])
def test_non_finite_sample_is_refused_wherever_it_is(n, at):
    x = synth.random_walk(n, 3)
    x[at] = np.inf
    with pytest.raises(dtws.DtwsError) as e:
        dtws.Index(x)
    assert e.value.status == dtws.DTWS_ENONFINITE


@pytest.mark.parametrize("n", [1024, 8192, 8197, 20001])
@pytest.mark.parametrize("m", [2, 3, 5, 6, 511, 1022, 1024])
def test_statistics_of_every_remainder(n, m):
    """Two windows a thread, every fourth window kept: every remainder of m and of
    the window count by four, windows that end with a block and with the series."""
    x = synth.random_walk(n, 80 + n + m)
    with dtws.Index(x) as ix:
        mh, ml, inv = ix.window_stats(m)
    mu, sg = oracle.window_stats(x, m, "twopass")
    got = mh.astype(np.float64) + ml.astype(np.float64)
    nz = sg > 0.0
    np.testing.assert_array_equal(inv == 0.0, ~nz)
    assert np.all(np.abs(got[nz] - mu[nz]) <= 1e-7 * sg[nz] + 1e-12 * np.abs(mu[nz]))
    assert np.abs(inv[nz].astype(np.float64) * sg[nz] - 1.0).max() <= 2.0 ** -22


@pytest.mark.parametrize("n", [2, 4095, 4097, 20_003])
@pytest.mark.parametrize("r", [0, 1, 2, 3, 4, 5, 6, 7, 9, 16, 31, 100, 1023, 4096, 8191])
def test_envelope_of_every_remainder(n, r):
    """The group split at every remainder of r, tiles past the series' end."""
    x = synth.random_walk(n, 90 + n)
    with dtws.Index(x) as ix:
        U, L = ix.series_envelope(r)
    Uo, Lo = oracle.series_envelope(x, r)
    np.testing.assert_array_equal(U, Uo)
    np.testing.assert_array_equal(L, Lo)
