"""Calls at the limits of what the entry points accept: thresholds that the line
pass rejects, several host threads, the longest series and the largest
minibatches."""
import numpy as np
import pytest

from oracle import c_oracle as CO
from oracle import rqa_oracle as O

pytestmark = pytest.mark.gpu


def _sine(n, period=628.0):
    return np.sin(2 * np.pi * np.arange(n) / period).astype(np.float32)


# Rows are cut into chunks from Ne = 257 on, and a second kernel joins the lines
# at the cuts.  A series with rejected thresholds has none; its neighbours keep
# theirs, whatever an earlier call left in the scratch.
@pytest.mark.parametrize("bad", [[0.5, 0.2], [-0.5, 0.2], [0.2, np.nan]])
@pytest.mark.parametrize("vertical,schedule", [(False, 0), (False, 1), (True, 0)])
def test_rejected_thresholds_beside_valid_ones(rqa_lib, vertical, schedule, bad):
    import torch
    rqa = rqa_lib
    ctx = rqa.Context(select=rqa.RQA_SELECT_RADIX, schedule=schedule)

    def lines(ys, eps):
        batch = rqa.Batch.from_numpy(ys, 1, 1)
        e = torch.tensor(eps, dtype=torch.float32, device="cuda")
        if vertical:
            out = rqa.vline_hist(ctx, batch, e, 2)
            out = {"hist": out["vhist"], "hist_offsets": out["vhist_offsets"], "lmax": out["vmax"], "count": out["vmass"]}
        else:
            out = rqa.line_hist(ctx, batch, e, 2)
        code = rqa.rqa_status(ctx)
        hist = rqa.unpack_hist(out["hist"].cpu().numpy(), out["hist_offsets"], batch, 2)
        return code, hist, out["lmax"].cpu().numpy(), out["count"].cpu().numpy()

    assert lines([_sine(3000)], [[0.1, 3.0]])[0] == 0  # long lines over every cut
    good = [0.2, 0.5]
    ys = [_sine(300), _sine(310), _sine(800)]
    code, hist, lmax, count = lines(ys, [bad, good, bad])
    assert code == 8
    if vertical:
        ref = O.vline_hist(ys[1], 1, 1, good)
        assert np.array_equal(hist[1], ref["vhist"]) and np.array_equal(lmax[1], ref["vmax"])
    else:
        ref = CO.lines(ys[1], 1, 1, good)
        assert np.array_equal(hist[1], ref["hist"]) and np.array_equal(lmax[1], ref["lmax"])
        assert np.array_equal(count[1], ref["count"])
    for s in (0, 2):
        assert not hist[s].any() and not lmax[s].any() and not count[s].any(), s
    ctx.close()


# The longest series that are accepted: the walks look up to 158 values past the
# end, so their indexes pass 2^31.  The same vectors stored without gaps are the
# reference (m windows of Ne values, one after the other).  m: a window per
# coordinate, rows of the line pass, values through L1.
@pytest.mark.parametrize("m", [2, 5, 9])
def test_longest_series(rqa_lib, m):
    import torch
    rqa = rqa_lib
    n = (1 << 31) - 65
    tau = (n - 300) // (m - 1)
    ne = n - (m - 1) * tau
    rng = np.random.default_rng(m)
    z = rng.standard_normal(m * ne).astype(np.float32)
    y = torch.zeros(n, dtype=torch.float32, device="cuda")
    for q in range(m):
        y[q * tau:q * tau + ne] = torch.from_numpy(z[q * ne:(q + 1) * ne]).cuda()
    batch = rqa.Batch(y, np.array([0, n]), m, tau)
    rr = [5, 30, 70]
    ctx = rqa.Context(select=rqa.RQA_SELECT_RADIX)
    sel = rqa.eps_for_rr(ctx, batch, rr, 100)
    lines = rqa.line_hist(ctx, batch, sel["eps"], 3)
    vert = rqa.vline_hist(ctx, batch, sel["eps"], 3)
    grid = rqa.eps_approx(ctx, batch, rr, 100, 40)
    assert rqa.rqa_status(ctx) == 0
    ref = O.eps_for_rr(z, m, ne, rr, 100)
    assert np.array_equal(sel["eps"].cpu().numpy()[0], ref["eps"])
    assert np.array_equal(sel["count_le"].cpu().numpy()[0], ref["count_le"])
    hist = CO.lines(z, m, ne, ref["eps"])["hist"]
    assert np.array_equal(lines["hist"].cpu().numpy().reshape(3, -1), hist)
    vhist = O.vline_hist(z, m, ne, ref["eps"])["vhist"]
    assert np.array_equal(vert["vhist"].cpu().numpy().reshape(3, -1), vhist)
    approx = O.eps_approx(z, m, ne, rr, 100, 40)
    assert np.array_equal(grid["eps"].cpu().numpy()[0], approx["eps"])
    assert np.array_equal(grid["count"].cpu().numpy()[0], approx["count"])
    ctx.close()


# One context per host thread: calls of different sizes, whose kernels take
# different amounts of shared memory, at the same time.  The kernels of these
# pairs differ in nothing else: short-series selection by the longest series,
# the middle counting round by the targets, the grid count by the thresholds.
@pytest.mark.parametrize("call", ["short", "middle", "grid"])
def test_threads_with_calls_of_different_sizes(rqa_lib, call):
    import threading

    import torch
    rqa = rqa_lib
    rng = np.random.default_rng(5)
    small, large = {"short": (100, 512), "middle": (25, 48), "grid": (8, 1024)}[call]
    errors = []

    def work(size, passes):
        try:
            n = size if call == "short" else 600
            y = rng.standard_normal(2 * n).astype(np.float32)
            stream = torch.cuda.Stream()
            with torch.cuda.stream(stream):
                ctx = rqa.Context(stream=stream, select=rqa.RQA_SELECT_RADIX)
                batch = rqa.Batch.from_numpy([y], 2, n)
                rr = list(range(1, 1 + (size if call == "middle" else 20)))
                outs = []
                for i in range(passes):
                    if call == "grid":
                        out = rqa.eps_approx(ctx, batch, rr, 100, size)
                    else:
                        out = rqa.eps_for_rr(ctx, batch, rr, 100)
                    if i in (0, passes - 1):
                        outs.append(out["eps"].clone())
                assert rqa.rqa_status(ctx) == 0
                assert torch.equal(outs[0], outs[1])
                ctx.close()
        except Exception as e:  # noqa: BLE001 - handed to the test's thread
            errors.append((size, repr(e)))

    threads = [threading.Thread(target=work, args=(size, 3000)) for size in (small, large)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors


def test_network_on_millions_of_rows(rqa_lib):
    """More rows than 65535 tiles of 32: nine rows repeated.  A row's outputs do
    not depend on the others, so they are the small batch's bit for bit; the
    gradients are means over the rows, so the small batch's but for rounding."""
    import torch
    rqa = rqa_lib
    rep = 233017
    B = 9 * rep  # 2097153
    g = torch.Generator(device="cuda").manual_seed(4)
    p = 0.05 * torch.randn(rqa.RQA_MLP_PARAMS, device="cuda", generator=g)
    x = torch.randn((9, 131), device="cuda", generator=g)
    t = torch.randn((9, 20), device="cuda", generator=g)
    ctx = rqa.Context()

    def run(X, T):
        n = X.shape[0]
        Y = torch.empty((n, 40), device="cuda")
        acts = torch.empty(n * 512, device="cuda")
        grads = torch.empty_like(p)
        rqa.rqa_mlp_forward(ctx, p, X, Y, acts.view(n, 512))
        rqa.rqa_mlp_backward(ctx, p, X, acts.view(n, 512), Y, T, 0.05, 0.95, grads)
        return Y, acts, grads

    Y, acts, grads = run(x.repeat(rep, 1), t.repeat(rep, 1))
    y, a, _ = run(x, t)
    assert rqa.rqa_status(ctx) == 0
    assert torch.equal(Y, y.repeat(rep, 1))
    for i in (0, 1):
        h = acts[i * B * 256:(i + 1) * B * 256].view(rep, 9, 256)
        assert torch.equal(h, a[i * 9 * 256:(i + 1) * 9 * 256].view(1, 9, 256).expand(rep, 9, 256))
    # the gradients in 64 bits and, with absolute values throughout, the scale of
    # their rounding: a sum of B rows by four partial sums is within
    # (B / 4 + 1000) 2^-24 < 0.04 of it
    W1, b1, W2, b2, W3, b3 = torch.split(p.double(), [256 * 131, 256, 256 * 256, 256, 40 * 256, 40])
    W1, W2, W3 = W1.view(256, 131), W2.view(256, 256), W3.view(40, 256)
    h1, h2 = a[:9 * 256].view(9, 256).double(), a[9 * 256:].view(9, 256).double()
    q = torch.tensor([0.05, 0.95], device="cuda").double().repeat(20)
    dY = torch.where(t.repeat_interleave(2, 1) >= y, -q, 1 - q) / (9 * 40)

    def chain(dY, W3, W2, x):
        dZ2 = (dY @ W3) * (h2 > 0)
        dZ1 = (dZ2 @ W2) * (h1 > 0)
        parts = (dZ1.T @ x, dZ1.sum(0), dZ2.T @ h1, dZ2.sum(0), dY.T @ h2, dY.sum(0))
        return torch.cat([v.reshape(-1) for v in parts])

    want = chain(dY, W3, W2, x.double())
    scale = chain(dY.abs(), W3.abs(), W2.abs(), x.double().abs())
    assert ((grads.double() - want).abs() <= 0.04 * scale).all()
    ctx.close()


def test_many_sizes_in_one_thread(rqa_lib):
    """More pairs of kernel and size than the launchers remember."""
    rqa = rqa_lib
    rng = np.random.default_rng(8)
    y = rng.standard_normal(600).astype(np.float32)
    ctx = rqa.Context(select=rqa.RQA_SELECT_RADIX)
    batch = rqa.Batch.from_numpy([y], 3, 1)
    for n_thr in list(range(1, 80)) + [40, 400]:
        out = rqa.eps_approx(ctx, batch, [10, 50], 100, n_thr)
        assert rqa.rqa_status(ctx) == 0
        ref = O.eps_approx(y, 3, 1, [10, 50], 100, n_thr)
        assert np.array_equal(out["eps"].cpu().numpy()[0], ref["eps"]), n_thr
        assert np.array_equal(out["count"].cpu().numpy()[0], ref["count"]), n_thr
    ctx.close()


@pytest.mark.parametrize("own_stream", [False, True])
def test_phase_times_without_a_graph(rqa_lib, own_stream):
    """Timing of calls that are not recorded in a graph (thresholds or lines
    alone, or any on the default stream)."""
    import torch
    rqa = rqa_lib
    stream = torch.cuda.Stream() if own_stream else torch.cuda.default_stream()
    with torch.cuda.stream(stream):
        ctx = rqa.Context(select=rqa.RQA_SELECT_RADIX, stream=stream)
        batch = rqa.Batch.from_numpy([_sine(3000)], 3, 1)
        rqa.rqa_set_timing(ctx, True)
        det = rqa.det_avg(ctx, batch, [5, 10], 100)
        assert rqa.rqa_status(ctx) == 0
        ms = rqa.rqa_phase_times(ctx)
        assert (ms[1:5] > 0).all()
        rqa.eps_for_rr(ctx, batch, [5, 10], 100)
        rqa.line_hist(ctx, batch, det["eps"], 2)
        assert rqa.rqa_status(ctx) == 0
        assert rqa.rqa_phase_times(ctx)[4] > 0
        ctx.close()
