"""The fixed-point re-score walk (up to two offsets per SM of dtws_dtw_at_f64,
the pre-score and the final stage of a search) against the FP64 oracle, at the
edges of its shapes: 32 K >= r + 2 cells for K = 1, 2, 3, 4 on one warp, 120 W
+ 8 >= r + 2 on W = 2, 3, 4, 6, 9, whole and ragged chunks of anti-diagonals,
its widest band and the first past it.

Tolerance: costs carry the double-float normalisation (2^-48 of |z| <= sqrt(m)
against differences of ~0.05 sigma and more: ~2^-40 per term at worst) and the
oracle's own FP64 sums; 1e-10 relative covers both with room."""
import numpy as np
import pytest

import oracle
from paper_1812_10302_gb300 import dtws, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def series():
    x = synth.random_walk(40_000, 15)
    x[3000:3600] = 7.25  # constant windows
    return x


@pytest.mark.parametrize("m,r", [(2, 0), (2, 1), (3, 2), (8, 7), (9, 3), (31, 30), (32, 31), (64, 31), (65, 62), (100, 63),
                                 (128, 94), (129, 95), (300, 126), (301, 127), (400, 190), (401, 191), (600, 254),
                                 (600, 255), (1000, 100), (5000, 30), (8192, 20), (8192, 254)])
def test_at_the_edges_of_its_shapes(series, m, r):
    q, o = synth.noisy_copy(series, m, m + r, m + 2 * r, noise=0.1)
    offs = np.random.default_rng(m + r).integers(0, series.size - m + 1, 24)
    offs[:3] = [o, 0, series.size - m]
    if m <= 600:
        offs[3] = 3000
    with dtws.Index(series) as ix:
        got = ix.dtw_at_f64(q, r, offs)
        assert ix.sync_status() == dtws.DTWS_OK
    want = oracle.dtw_at(series, q, r, offs)
    np.testing.assert_allclose(got, want, rtol=1e-10, atol=1e-18 * m)


@pytest.mark.parametrize("m,r", [(127, 126), (128, 127), (247, 246), (248, 247), (500, 246), (501, 247), (367, 366),
                                 (700, 367), (487, 486), (990, 487), (727, 726), (801, 727), (1023, 1022),
                                 (1025, 1023), (1100, 1024)])
def test_several_walking_warps(series, m, r):
    """Bands past one warp: the overlaps of two to nine warps, each at its widest
    band and the first past it, queries no longer than the band and longer,
    both parities of m + r (where the walks from both ends meet)."""
    q, o = synth.noisy_copy(series, m, m + r, m + 2 * r, noise=0.1)
    offs = np.random.default_rng(m + r).integers(0, series.size - m + 1, 5)
    offs[:3] = [o, 0, series.size - m]
    with dtws.Index(series) as ix:
        got = ix.dtw_at_f64(q, r, offs)
        idx, dist = ix.query(q, r, 2)
        assert ix.sync_status() == dtws.DTWS_OK
    np.testing.assert_allclose(got, oracle.dtw_at(series, q, r, offs), rtol=1e-10)
    oi, od = oracle.search_cascade(series, q, r, 2)
    np.testing.assert_array_equal(idx, oi)
    np.testing.assert_allclose(dist, od, rtol=1e-6)


@pytest.mark.parametrize("m,r", [(500, 487), (620, 600), (740, 730), (1060, 1000)])
def test_clusters_of_four_in_several_waves(series, m, r):
    """Bands whose costs come from a second pair of CTAs (six and nine walking
    warps), with twice as many clusters as fit the GPU: a cluster of a later
    wave starts, CTA by CTA, as earlier ones end, and none of its CTAs touches
    another's shared memory before all have started."""
    q, o = synth.noisy_copy(series, m, m + r, m + 2 * r, noise=0.1)
    offs = np.random.default_rng(m + r).integers(0, series.size - m + 1, 70)
    offs[:3] = [o, 0, series.size - m]
    with dtws.Index(series) as ix:
        got = [ix.dtw_at_f64(q, r, offs) for _ in range(5)]
        assert ix.sync_status() == dtws.DTWS_OK
    np.testing.assert_allclose(got[0], oracle.dtw_at(series, q, r, offs), rtol=1e-10)
    for g in got[1:]:
        np.testing.assert_array_equal(g, got[0])


@pytest.mark.parametrize("unnormalised,scale", [(0, 1.0), (1, 1.0), (1, 2.0 ** -30), (1, 2.0 ** 20)])
def test_far_below_the_euclidean_distance(unnormalised, scale):
    """Shifted copies of a smooth window: warping absorbs the shift, so the DTW
    lies orders of magnitude below the bound that first scales the walk, which
    is then repeated on a finer scale."""
    t = np.arange(6000)
    x = ((np.sin(t / 40.0) + 0.3 * np.sin(t / 17.0 + 1.0)) * 100.0 * scale).astype(np.float32)
    m, r = 512, 60
    q = x[1000:1000 + m].copy()
    offs = np.array([1000, 1001, 1003, 1010, 1030, 1055, 900, 2500])
    with dtws.Index(x, options=dict(unnormalised=unnormalised)) as ix:
        got = ix.dtw_at_f64(q, r, offs)
        assert ix.sync_status() == dtws.DTWS_OK
    want = (np.array([oracle.dtw(q, x[o:o + m], r) for o in offs]) if unnormalised
            else oracle.dtw_at(x, q, r, offs))
    assert got[0] <= 1e-20 * want[-1]
    np.testing.assert_allclose(got[1:], want[1:], rtol=1e-8)


def test_a_match_and_its_exact_copies_keep_their_order():
    """The pre-scored window and later bit-identical copies of it come back in
    offset order: compared windows are walked with one bound."""
    x = synth.random_walk(30_000, 77)
    m = 200
    for at in (20_000, 9_000, 25_000):
        x[at:at + m] = x[4_000:4_000 + m]
    q = x[4_000:4_000 + m] + np.random.default_rng(5).normal(0, 0.05, m).astype(np.float32)
    with dtws.Index(x) as ix:
        for k in (1, 4):
            idx, dist = ix.query(q, 20, k)
            np.testing.assert_array_equal(idx, [4_000, 9_000, 20_000, 25_000][:k])
            assert np.all(dist == dist[0])


@pytest.mark.parametrize("m,r", [(2, 0), (2, 1), (3, 1), (9, 8), (40, 22), (41, 23), (60, 38), (60, 39), (100, 46), (101, 47),
                                 (101, 54), (102, 55), (200, 78), (201, 79), (200, 94), (200, 95), (300, 110), (301, 111),
                                 (300, 158), (300, 159), (400, 222), (401, 223), (2500, 20)])
def test_many_offsets(series, m, r):
    """The throughput shapes (more than two offsets per SM) at their widest bands
    and the first past them, both parities, constant and repeated windows, a
    spike that sets the grid the values are split on."""
    x = series.copy()
    x[9000] += 1e4
    q, o = synth.noisy_copy(x, m, m + r, m + 2 * r, noise=0.1)
    some = np.random.default_rng(m + r).integers(0, x.size - m + 1, 24)
    some[:5] = [o, 0, x.size - m, 3000, 9000 - m // 2]
    offs = np.tile(some, 14)
    with dtws.Index(x) as ix:
        got = ix.dtw_at_f64(q, r, offs)
        few = ix.dtw_at_f64(q, r, some)
        assert ix.sync_status() == dtws.DTWS_OK
    want = oracle.dtw_at(x, q, r, some)
    np.testing.assert_allclose(got[:24], want, rtol=1e-10, atol=1e-18 * m)
    np.testing.assert_array_equal(got, np.tile(got[:24], 14))
    np.testing.assert_allclose(few, want, rtol=1e-10, atol=1e-18 * m)


@pytest.mark.parametrize("m,r", [(60, 23), (200, 78), (400, 222)])
@pytest.mark.parametrize("power", [-60, -27, 100, 118, None])
def test_many_offsets_in_any_units(series, m, r, power):
    """The throughput shapes on a series times a power of two (None: the largest
    that FP32 holds, both signs among the samples of a window): normalisation
    takes the units off exactly, so the distances are those of the plain series,
    as those of few offsets are.  (Below 2^-27 no window's variance may fall
    under the zero-variance rule's 1e-24: constant windows are left out.)"""
    x = (series - np.float32(7.25)).astype(np.float32)
    x[::2] *= -1.0
    s = 127 - int(np.floor(np.log2(np.abs(x).max()))) if power is None else power
    q, o = synth.noisy_copy(x, m, m + r, m + 2 * r, noise=0.1)
    some = np.random.default_rng(m + r).integers(4000, x.size - m + 1, 24)
    some[:3] = [o, 0, x.size - m]
    xs, qs = np.ldexp(x, s), np.ldexp(q, s)
    assert np.isfinite(xs).all() and np.isfinite(qs).all()
    with dtws.Index(xs) as ix:
        many = ix.dtw_at_f64(qs, r, np.tile(some, 14))
        few = ix.dtw_at_f64(qs, r, some)
        assert ix.sync_status() == dtws.DTWS_OK
    want = oracle.dtw_at(x, q, r, some)
    if power == -60:  # sigma ~ 1e-17: every window counts as constant, the query too
        np.testing.assert_array_equal(many, np.zeros(many.size))
        np.testing.assert_array_equal(few, np.zeros(few.size))
        return
    np.testing.assert_allclose(few, want, rtol=1e-10)
    np.testing.assert_allclose(many, np.tile(want, 14), rtol=1e-10)
