"""DTW at given offsets in the shapes for many windows (lanes x cells per lane)
at the bands where the shape changes, through the handle and without
allocations, against the FP64 oracle: FP32 walks of at most 2 m squared terms,
1e-4 relative as for every FP32 distance of the library."""
import numpy as np
import pytest

import oracle
from paper_1812_10302_gb300 import dtws, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def series():
    x = synth.random_walk(25_000, 45)
    x[7000:7400] = -3.0  # constant windows
    return x


@pytest.mark.parametrize("m,r", [(2, 1), (5, 4), (40, 3), (40, 4), (40, 5), (64, 6), (64, 7), (64, 8), (65, 9), (90, 10),
                                 (100, 12), (100, 13), (128, 18), (128, 19), (129, 22), (200, 26), (200, 27), (300, 30),
                                 (300, 38), (301, 54), (301, 55), (400, 62), (400, 78), (500, 110), (500, 111),
                                 (600, 126), (600, 158), (600, 159), (700, 222), (700, 254), (700, 255), (700, 256),
                                 (3000, 5), (4096, 40), (8192, 12), (8192, 254)])
@pytest.mark.parametrize("count", [1, 45])
def test_at_shape_edges(series, m, r, count):
    import torch
    q, _ = synth.noisy_copy(series, m, 2 * m + r, m + 7, noise=0.3)
    offs = np.random.default_rng(m * r + count).integers(0, series.size - m + 1, count)
    offs[-1] = series.size - m
    if count > 3:
        offs[:3] = [0, min(7000, series.size - m), offs[4]]
    want = oracle.dtw_at(series, q, r, offs)
    with dtws.Index(series) as ix:
        got = ix.dtw_at(q, r, offs)
        many = ix.dtw_at(q, r, np.tile(offs, 40))
    np.testing.assert_allclose(got, want, rtol=1e-4, atol=1e-6 * m)
    np.testing.assert_array_equal(many, np.tile(got, 40))
    xs, qs, os_ = (torch.from_numpy(a).cuda() for a in (series, q, offs))
    out = torch.empty(count, device="cuda")
    st = dtws.load().dtws_dtw_at_noalloc(xs.data_ptr(), series.size, qs.data_ptr(), m, r, os_.data_ptr(), count,
                                         out.data_ptr(), torch.cuda.current_stream().cuda_stream)
    assert st == dtws.DTWS_OK
    np.testing.assert_allclose(out.cpu().numpy(), want, rtol=1e-4, atol=1e-6 * m)


def test_bad_device_offsets_give_nan(series):
    import torch
    q, _ = synth.noisy_copy(series, 128, 3, 4, noise=0.3)
    offs = torch.tensor([5, -1, series.size - 127, 77, 2 ** 40], device="cuda")
    with dtws.Index(series) as ix:
        for r in (2, 12, 100):
            got = ix.dtw_at(q, r, offs)
            np.testing.assert_array_equal(np.isnan(got), [False, True, True, False, True])


@pytest.mark.parametrize("scale", [1e-8, 1e30, 3e35])
def test_without_allocations_in_any_units(series, scale):
    """Values whose squares, and sums, leave FP32's range: normalisation takes
    the units off, so the distances are those of the series in plain units
    (each value off by an ulp of itself, as in the 1e-4 above)."""
    import torch
    q, _ = synth.noisy_copy(series, 128, 9, 11, noise=0.3)
    offs = np.random.default_rng(3).integers(0, series.size - 127, 40)
    xs = (series.astype(np.float64) * scale).astype(np.float32)
    qs = (q.astype(np.float64) * scale).astype(np.float32)
    assert np.isfinite(xs).all()
    for r in (3, 12):
        want = oracle.dtw_at(xs.astype(np.float64) / scale, qs.astype(np.float64) / scale, r, offs)
        xd, qd, od = (torch.from_numpy(a).cuda() for a in (xs, qs, offs))
        out = torch.empty(offs.size, device="cuda")
        st = dtws.load().dtws_dtw_at_noalloc(xd.data_ptr(), series.size, qd.data_ptr(), 128, r, od.data_ptr(),
                                             offs.size, out.data_ptr(), torch.cuda.current_stream().cuda_stream)
        assert st == dtws.DTWS_OK
        np.testing.assert_allclose(out.cpu().numpy(), want, rtol=1e-4, atol=1e-6 * 128)
