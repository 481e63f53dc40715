"""How the cell passes split their work: short series selected by one CTA each,
rows cut into chunks whose lines are joined afterwards, ranges of keys that are
counted densely or through tables, windows per coordinate.  Sizes lie at the
edges of these splits; everything is compared with the oracle, bit for bit."""
import numpy as np
import pytest

from oracle import rqa_oracle as O
from tests._helpers import RR20, assert_series_equal, gpu_run, oracle_series
from tests.test_gpu_vlines import _check as check_vertical

pytestmark = pytest.mark.gpu


def _compare(ys, m, tau, rr, schedules=(0, 1), lmin=(1, 2, 5)):
    """m and tau: one for all series or one per series."""
    ms, taus = np.broadcast_to(m, len(ys)), np.broadcast_to(tau, len(ys))
    refs = [oracle_series(y, int(a), int(b), rr, 100, lmin=lmin) for y, a, b in zip(ys, ms, taus)]
    for schedule in schedules:
        g = gpu_run(ys, m, tau, rr, 100, lmin=lmin, schedule=schedule)
        for s, ref in enumerate(refs):
            assert_series_equal(g, s, ref, f"m={ms[s]} tau={taus[s]} n={len(ys[s])} schedule {schedule}")


# Ne of the short-series path ends at 512, its samples at 1024, its targets at 24
@pytest.mark.parametrize("K", [1, 24, 25])
@pytest.mark.parametrize("ne,m,tau", [(2, 1, 1), (33, 3, 1), (511, 2, 3), (512, 3, 256), (513, 1, 1),
                                      (512, 2, 513)])
def test_short_series_selection(rqa_lib, ne, m, tau, K):
    rng = np.random.default_rng(ne * 31 + m + K)
    n = ne + (m - 1) * tau
    ys = [rng.standard_normal(n).astype(np.float32), rng.integers(0, 4, n).astype(np.float32),
          np.full(n, -2.5, np.float32), np.exp(8 * rng.standard_normal(n)).astype(np.float32)]
    _compare(ys, m, tau, list(range(2, 2 + K)), schedules=(0,))


def test_short_series_selection_reports_nonfinite(rqa_lib):
    rqa = rqa_lib
    for bad in (np.nan, np.inf):
        ys = [np.arange(40, dtype=np.float32), np.arange(50, dtype=np.float32)]
        ys[1][49] = bad
        ctx = rqa.Context(select=rqa.RQA_SELECT_RADIX)
        batch = rqa.Batch.from_numpy(ys, 1, 1)
        rqa.eps_for_rr(ctx, batch, RR20, 100)
        assert rqa.rqa_status(ctx) == 3  # a series holds NaN or an infinity
        ctx.close()


def _long_lines(n, seed):
    """Lines that cross many rows, short ones, one for each diagonal."""
    rng = np.random.default_rng(seed)
    t = np.arange(n)
    x = np.sin(2 * np.pi * t / 20.3)
    x[n // 2:n // 2 + 2] += 3  # a break, so that lines end in the middle too
    return [x.astype(np.float32), rng.standard_normal(n).astype(np.float32), np.full(n, 0.5, np.float32)]


# rows are cut at multiples of 32 from 256 on; one series and few targets per
# launch, so that the series is cut as finely as it can be
@pytest.mark.parametrize("m,tau", [(1, 1), (3, 1), (3, 3), (2, 2), (4, 2), (5, 1)])
@pytest.mark.parametrize("ne", [255, 257, 513, 1025])
def test_rows_in_chunks(rqa_lib, ne, m, tau):
    ys = _long_lines(ne + (m - 1) * tau, ne + m)
    _compare(ys, m, tau, [1, 5, 20, 60, 95], schedules=(1,))
    _compare(ys[:2], m, tau, RR20, schedules=(0,))


@pytest.mark.parametrize("m,tau", [(1, 1), (3, 3), (4, 2), (5, 1)])
@pytest.mark.parametrize("ne", [257, 513, 769])
def test_rows_in_chunks_vertical(rqa_lib, ne, m, tau):
    check_vertical(rqa_lib, _long_lines(ne + (m - 1) * tau, ne - m), m, tau, [1, 5, 20, 60, 95], 1, False)
    check_vertical(rqa_lib, _long_lines(ne + (m - 1) * tau, ne - m)[:2], m, tau, RR20, 0, True)


# targets that fall into few, many and widely spread ranges of keys
@pytest.mark.parametrize("rr", [[50], RR20, list(range(1, 100))])
@pytest.mark.parametrize("m,tau", [(1, 1), (3, 1), (2, 5)])
def test_counted_ranges(rqa_lib, m, tau, rr):
    rng = np.random.default_rng(len(rr) + m)
    n = 700
    ys = [rng.standard_normal(n).astype(np.float32),
          rng.integers(0, 50, n).astype(np.float32) / 8,
          np.exp(12 * rng.standard_normal(n)).clip(1e-30, 1e30).astype(np.float32),
          (1e-38 * rng.standard_normal(n)).astype(np.float32),  # denormal distances
          np.concatenate([np.zeros(n - 20), rng.standard_normal(20)]).astype(np.float32)]
    _compare(ys, m, tau, rr)


# windows per coordinate for m <= 8, samples through L1 above it; Ne around the
# 28-row blocks and 128-diagonal bands
@pytest.mark.parametrize("m_max", [6, 7, 8, 9])
def test_mixed_embeddings(rqa_lib, m_max):
    rng = np.random.default_rng(m_max)
    ys, ms, taus = [], [], []
    for i, ne in enumerate([2, 27, 28, 29, 57, 127, 128, 129, 130, 257, 561]):
        m, tau = (m_max - i) % m_max + 1, (3 * i) % 5 + 1
        ys.append(rng.standard_normal(ne + (m - 1) * tau).astype(np.float32))
        ms.append(m)
        taus.append(tau)
    assert max(ms) == m_max
    _compare(ys, np.array(ms), np.array(taus), list(range(3, 93, 3)))


# grids that one multiplication locates, and grids whose steps are lost in the
# type's smallest values or overflow, which are searched
@pytest.mark.parametrize("scale", [1e-42, 1e-38, 1e-20, 1.0, 1e30])
@pytest.mark.parametrize("m,tau,n_thr", [(1, 1, 1024), (3, 3, 400), (2, 2, 1), (6, 1, 33), (7, 2, 100), (8, 2, 100), (9, 1, 50)])
def test_grid_of_any_scale(rqa_lib, scale, m, tau, n_thr):
    rqa = rqa_lib
    rng = np.random.default_rng(n_thr)
    ys = [(scale * rng.standard_normal(300)).astype(np.float32), np.full(290, scale, np.float32),
          (scale * rng.integers(0, 9, 400)).astype(np.float32)]
    rr = [1, 7, 30, 88]
    ctx = rqa.Context(select=rqa.RQA_SELECT_RADIX)
    batch = rqa.Batch.from_numpy(ys, m, tau)
    g = rqa.eps_approx(ctx, batch, rr, 100, n_thr)
    assert rqa.rqa_status(ctx) == 0
    eps, rate, cnt = (g[k].cpu().numpy() for k in ("eps", "rr", "count"))
    for s, y in enumerate(ys):
        ref = O.eps_approx(y, m, tau, rr, 100, n_thr)
        assert np.array_equal(eps[s], ref["eps"]), s
        assert np.array_equal(rate[s], ref["rr"]), s
        assert np.array_equal(cnt[s], ref["count"]), s
    ctx.close()
