"""Row chunks of the line pass and the joining of their lines: batches of unlike
lengths (some series cut, most not), several target groups, lines over 44 and 64
cells, tuned units, and the sizes at which a batch is cut at all.  Everything is
compared with the oracle, bit for bit."""
import numpy as np
import pytest

from oracle import c_oracle as CO
from oracle import rqa_oracle as O
from tests._helpers import RR20

pytestmark = pytest.mark.gpu


def _wave(n, seed):
    """Long lines with breaks at every scale."""
    rng = np.random.default_rng(seed)
    x = np.sin(2 * np.pi * np.arange(n) / 31.7) + 0.02 * rng.standard_normal(n)
    x[rng.integers(0, n, 2 + n // 300)] += 1.5
    return x.astype(np.float32)


def _check(rqa, ys, m, tau, rr, tuning=None, vertical=False, schedule=0):
    """ys may repeat an array: its oracle is worked out once."""
    K = len(rr)
    ctx = rqa.Context(select=rqa.RQA_SELECT_RADIX, schedule=schedule)
    if tuning:
        rqa.rqa_set_tuning(ctx, **tuning)
    batch = rqa.Batch.from_numpy(ys, m, tau)
    sel = rqa.eps_for_rr(ctx, batch, rr, 100)
    if vertical:
        out = rqa.vline_hist(ctx, batch, sel["eps"], K)
        hist, off, lmax, count = out["vhist"], out["vhist_offsets"], out["vmax"], out["vmass"]
    else:
        out = rqa.line_hist(ctx, batch, sel["eps"], K)
        hist, off, lmax, count = out["hist"], out["hist_offsets"], out["lmax"], out["count"]
    assert rqa.rqa_status(ctx) == 0
    eps, le = sel["eps"].cpu().numpy(), sel["count_le"].cpu().numpy()
    hist, lmax, count = (t.cpu().numpy() for t in (hist, lmax, count))
    refs = {}
    for s, y in enumerate(ys):
        if id(y) not in refs:
            ref = O.vline_hist(y, m, tau, eps[s]) if vertical else CO.lines(y, m, tau, eps[s])
            refs[id(y)] = (ref["vhist"], ref["vmax"]) if vertical else (ref["hist"], ref["lmax"])
        h, longest = refs[id(y)]
        assert np.array_equal(hist[off[s]:off[s + 1]].reshape(K, -1), h), s
        assert np.array_equal(lmax[s], longest), s
        assert np.array_equal(count[s], (2 if vertical else 1) * le[s]), s
    ctx.close()


# 700 series shorter than a chunk beside a few that are cut: the cut bands are
# shared among the joining kernel's CTAs whatever series they are of
@pytest.mark.parametrize("m,tau,rr", [(1, 1, RR20), (3, 3, [2, 40]), (3, 2, list(range(2, 92, 2)))])
def test_batch_of_unlike_lengths(rqa_lib, m, tau, rr):
    short = [_wave(n, n) for n in (40, 255, 257)]
    ys = [_wave(n, n) for n in (2500, 300, 601, 1111)] + [short[i % 3] for i in range(700)]
    _check(rqa_lib, ys, m, tau, rr)


def test_batch_of_unlike_lengths_vertical(rqa_lib):
    ys = [_wave(n, n) for n in (900, 40, 300, 256, 257)]
    _check(rqa_lib, ys, 2, 3, [3, 30, 60], vertical=True)


@pytest.mark.parametrize("schedule", [0, 1])
@pytest.mark.parametrize("unit_bands", [1, 3, 64])
def test_tuned_units_of_cut_bands(rqa_lib, unit_bands, schedule):
    ys = [_wave(n, n) for n in (1800, 290, 33, 700)]
    _check(rqa_lib, ys, 3, 1, RR20, tuning={"unit_bands": unit_bands, "line_ctas": 2}, schedule=schedule)


# Batches whose longest band has at most 32 blocks of 32 rows and no more than
# twice a warp's share stay whole: 130 series of 1024 (m = 1) do, of 1025 not
@pytest.mark.parametrize("n,copies", [(1024, 65), (1025, 65), (600, 30), (600, 100)])
def test_whole_and_cut_bands(rqa_lib, n, copies):
    a, b = _wave(n, 1), _wave(n, 2)
    _check(rqa_lib, [a, b] * copies, 1, 1, [4, 11, 35])
