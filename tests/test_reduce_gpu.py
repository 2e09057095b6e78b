"""aeb_reduce against its plain definition at the edges of its split (a warp, a
block's share, several blocks), of its histograms and of its values."""
import math

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def aeb():
    import paper_2604_27193_gb300 as m
    m.build()
    return m


@pytest.mark.parametrize("lo_d,lo_v", [(0.0, 0.0), (-3.0, 0.0), (0.0, 1.5), (41.3, 7.7)])
@pytest.mark.parametrize("n", [1, 31, 33, 2048, 2049, 70_001])
def test_reduction_at_its_edges(aeb, n, lo_d, lo_v):
    """Sizes around a warp, a block's share and more blocks than one, histogram
    origins at and off zero, every status, and values that are zero, negative,
    tiny or huge: counts, bins and extremes exact, sums as accurate as n
    additions in binary64."""
    rng = np.random.default_rng(n)
    status = rng.choice(np.array([0, 1, 2, 255], np.uint8), n, p=[0.45, 0.45, 0.05, 0.05])
    x = rng.normal(40.0, 15.0, n)
    v = rng.uniform(0.0, 30.0, n)
    for a in (x, v):
        a[::17] = rng.choice([0.0, -0.0, -2.5, 1e-310, 5e3, 1e-3], len(a[::17]))
    steps = rng.integers(0, 10_000, n).astype(np.int32)
    out = {"status": torch.from_numpy(status).cuda(), "x_ref": torch.from_numpy(x).cuda(),
           "v_imp": torch.from_numpy(v).cuda(), "n_steps": torch.from_numpy(steps).cuda()}
    S = aeb.alloc_stats()
    h = aeb.hist_spec(lo_d=lo_d, lo_v=lo_v)
    aeb.aeb_reduce(out, n, h, S)
    st = aeb.stats_from_buffer(S)
    assert (st.n, st.steps) == (n, int(steps.sum()))
    assert [st.n_stop, st.n_contact, st.n_horizon, st.n_invalid] == [
        int((status == k).sum()) for k in (0, 1, 2, 255)]
    for a, lo, w, hist, s1, s2, mn, mx in (
            (x[status == 0], lo_d, h.w_d, st.hist_d, st.sum_d, st.sumsq_d, st.min_d, st.max_d),
            (v[status == 1], lo_v, h.w_v, st.hist_v, st.sum_v, st.sumsq_v, st.min_v, st.max_v)):
        b = np.clip(np.floor((a - lo) / w), 0, aeb.NBINS - 1).astype(int)
        assert np.array_equal(np.array(hist, np.int64), np.bincount(b, minlength=aeb.NBINS))
        assert mn == (a.min() if len(a) else math.inf) and mx == (a.max() if len(a) else -math.inf)
        assert abs(s1 - math.fsum(a)) <= n * 2.0 ** -52 * math.fsum(np.abs(a))
        assert abs(s2 - math.fsum(a * a)) <= (n + 1) * 2.0 ** -52 * math.fsum(a * a)
