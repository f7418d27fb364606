"""Searches whose queries match nothing, so that most windows are walked or
pruned late: the survivor pass's pre-check, lane by lane (long series) and by
whole groups, against the distance of every window (DTW at offsets, itself
held to the FP64 oracle)."""
import numpy as np
import pytest

from paper_1812_10302_gb300 import dtws, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def series():
    import torch
    return torch.from_numpy(synth.walk_with_bursts(1_500_000, 31, 32, 33)).cuda()


@pytest.mark.parametrize("m,r", [(3, 1), (10, 2), (65, 6), (66, 7), (67, 5), (100, 60), (129, 13), (130, 40), (131, 3), (300, 31),
                                 (257, 65)])
@pytest.mark.parametrize("n", [1_500_000, 40_000])
@pytest.mark.parametrize("exact_envelope", [0, 1])
def test_loose_queries(series, m, r, n, exact_envelope):
    """Query lengths around the 64 terms that the scan takes and the 128 that
    the pre-check takes, with and without the exact envelope of the series;
    a white-noise query, like no window of a walk, as tight as its best match."""
    import torch
    x = series[:n]
    q = torch.from_numpy(np.random.default_rng(m + n).standard_normal(m).astype(np.float32)).cuda()
    offs = torch.arange(n - m + 1, device="cuda")
    k = 3
    with dtws.Index(x, options=dict(exact_envelope=exact_envelope, seed_proposals=16 if exact_envelope else 0)) as ix:
        idx, dist = ix.query(q, r, k)
        assert ix.sync_status() in ((dtws.DTWS_OK, dtws.DTWS_EOVERFLOW) if m < 8 else (dtws.DTWS_OK,))
        d = ix.dtw_at(q, r, offs)
    best = np.sort(d)[:k]
    # both are FP32 walks of one window (1e-4) or their FP64 re-score
    np.testing.assert_allclose(dist, best, rtol=2e-4, atol=2e-6 * m)
    np.testing.assert_allclose(d[idx], dist, rtol=2e-4, atol=2e-6 * m)
    assert np.unique(idx).size == k
