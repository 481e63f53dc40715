"""Performance cases of the averaged-RQA library, through its public entry points.

Sizes and options are those of the repository's workloads, tests and benchmark: the
logistic map at N = 100, the Lorenz quartet at N = 1e4, the uneven batch of 720, the
long series of the full form with the learned bracket, RR = 1..99 %, the generic
embeddings, caller-given thresholds, vertical lines, the grid search, the bracket
network's training step and training labels, and the selection that does not allocate.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

import paper_2208_09136_gb300 as rqa
from paper_2208_09136_gb300 import bracket

KINDS = ("sine", "logistic", "lorenz")
SNRS = (-20.0, -15.0, -10.0, -5.0, 0.0, 5.0, 10.0, 20.0)
SEG = 400  # samples of one independently started piece of a chaotic signal


# ---------------------------------------------------------------- cases
def _det(name, sizes, m, tau, signals="mix", K=20, den=100, lmin="2", lines=False, learned=False, kept=False):
    return {"name": name, "what": "det", "sizes": sizes, "m": m, "tau": tau, "signals": signals, "K": K,
            "den": den, "lmin": lmin, "lines": lines, "learned": learned, "kept": kept}


def listed():
    return [
        # the smallest call: one short series, no embedding (interactive use, scripts over many short calls)
        _det("one-short", "1x100", 1, 1, "logistic"),
        # one record per noise level with its line histograms: the plain method at the usual length
        _det("lorenz-1e4", "4x10000", 3, 3, "lorenz", lines=True),
        # a study's batch: three signals, eight noise levels, ten seeds, lengths 1e2, 1e3 and 1e4
        _det("batched-720", "240x100,240x1000,240x10000", 3, 1),
        # the full form as the benchmark runs it: long and uneven short series, learned bracket,
        # histograms, three minimal line lengths, buffers and stream kept by the caller
        _det("long-learned", "24x100000,200xlog100-10000", 3, 3, lmin="2,3,5", lines=True, learned=True, kept=True),
        # averaging over RR = 1..99 % (K = 99), the embedding's delay not one of the usual two
        _det("rr-1-to-99", "6xlog3001-4001", 3, 2, K=99),
        # thresholds alone for a batch of unlike embeddings (m = 1..6, delays 1..4), odd lengths
        {"name": "eps-mixed", "what": "eps", "sizes": "60xlog101-5001", "m": 0, "tau": 0, "signals": "mix",
         "K": 20, "den": 100},
        # caller-chosen thresholds: histograms, average line length and entropy of two-dimensional embeddings
        {"name": "lines-given", "what": "lines", "sizes": "3x7001", "m": 2, "tau": 1, "signals": "mix", "K": 5,
         "lmin": "2,4"},
        # vertical lines, laminarity and trapping time of the whole matrix
        {"name": "vertical-5e3", "what": "vlines", "sizes": "4x5000", "m": 3, "tau": 3, "signals": "mix", "K": 20,
         "vmin": "2,3"},
        # the approximate search on a grid of 400 thresholds, then DET at its thresholds
        {"name": "grid-400", "what": "grid", "sizes": "8xlog2000-6000", "m": 3, "tau": 1, "signals": "mix",
         "K": 20, "den": 100, "n_thr": 400},
        # one optimiser step of the bracket network on a minibatch
        {"name": "train-step", "what": "train", "rows": 256},
        # training labels and features of a slice of the training set (exact radix selection)
        {"name": "train-labels", "what": "labels", "sizes": "300xlog100-10000", "m": 3, "tau": 3, "signals": "mix"},
        # thresholds for a caller that cannot allocate
        {"name": "noalloc", "what": "noalloc", "sizes": "2x2003", "m": 2, "tau": 3, "signals": "mix", "K": 10,
         "den": 100},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    what = rng.choice(("short", "mid", "batch", "long", "rr", "eps", "lines", "vlines", "grid", "train", "labels",
                       "noalloc"))
    sig = rng.choice(("mix", "mix") + KINDS)
    m, tau = rng.choice(((1, 1), (2, 1), (2, 3), (3, 1), (3, 3), (3, 3), (3, 5), (4, 2), (5, 1)))
    lmin = rng.choice(("2", "2,3,5", "3", "2,10"))
    if what == "short":
        n = _log(rng, 40, 600)
        c = _det("", "%dx%d" % (rng.choice((1, 1, 2, 7)), n), m, tau, sig, lmin=lmin, lines=rng.random() < 0.5)
    elif what == "mid":
        c = _det("", "%dx%d" % (rng.choice((1, 3, 4)), _log(rng, 2000, 20000)), m, tau, sig,
                 K=rng.choice((5, 10, 20, 20, 30)), lmin=lmin, lines=rng.random() < 0.5)
    elif what == "batch":
        c = _det("", "%dxlog%d-%d" % (_log(rng, 20, 400), rng.choice((50, 100, 301)), _log(rng, 1000, 8000)), 3, tau,
                 sig, lmin=lmin, kept=rng.random() < 0.5)
    elif what == "long":
        c = _det("", "%dx%d,20xlog100-5000" % (rng.choice((1, 2, 3, 5)), _log(rng, 30000, 100000)), 3, 3, sig,
                 lmin=lmin, lines=True, learned=rng.random() < 0.6, kept=True)
    elif what == "rr":
        c = _det("", "%dxlog%d-%d" % (rng.choice((1, 2, 6)), 200, _log(rng, 500, 4000)), m, tau, sig,
                 K=rng.choice((33, 50, 99)), lmin=lmin)
    elif what == "eps":
        c = {"what": "eps", "sizes": "%dxlog101-%d" % (_log(rng, 1, 100), _log(rng, 500, 6000)), "m": 0, "tau": 0,
             "signals": sig, "K": rng.choice((1, 10, 20, 20, 40)), "den": 100}
    elif what == "lines":
        c = {"what": "lines", "sizes": "%dx%d" % (rng.choice((1, 3, 9)), _log(rng, 300, 9000)), "m": m, "tau": tau,
             "signals": sig, "K": rng.choice((1, 3, 5, 12, 20)), "lmin": lmin}
    elif what == "vlines":
        c = {"what": "vlines", "sizes": "%dx%d" % (rng.choice((1, 4)), _log(rng, 300, 6000)), "m": m, "tau": tau,
             "signals": sig, "K": rng.choice((5, 20, 20)), "vmin": lmin}
    elif what == "grid":
        c = {"what": "grid", "sizes": "%dx%d" % (rng.choice((1, 8)), _log(rng, 300, 8000)), "m": m, "tau": tau,
             "signals": sig, "K": 20, "den": 100, "n_thr": rng.choice((25, 100, 400, 400, 1000))}
    elif what == "train":
        c = {"what": "train", "rows": _log(rng, 32, 2048)}
    elif what == "labels":
        c = {"what": "labels", "sizes": "%dxlog100-%d" % (_log(rng, 20, 300), _log(rng, 1000, 10000)), "m": 3,
             "tau": 3, "signals": sig}
    else:
        c = {"what": "noalloc", "sizes": "%dx%d" % (rng.choice((1, 2, 4)), _log(rng, 60, 8000)), "m": m, "tau": tau,
             "signals": sig, "K": rng.choice((5, 10, 20, 31)), "den": 100}
    c.pop("name", None)
    return c


def _sizes(case):
    """Series lengths: 'SxN' and 'SxlogLO-HI' groups; they depend on the case alone."""
    rng = random.Random(case["sizes"])
    out = []
    for part in case["sizes"].split(","):
        s, n = part.split("x")
        if n.startswith("log"):
            lo, hi = (int(v) for v in n[3:].split("-"))
            out += [_log(rng, lo, hi) for _ in range(int(s))]
        else:
            out += [int(n)] * int(s)
    return out


def _embedding(case, sizes):
    if case["m"]:
        return [case["m"]] * len(sizes), [case["tau"]] * len(sizes)
    rng = random.Random(len(sizes))
    return [rng.randint(1, 6) for _ in sizes], [rng.randint(1, 4) for _ in sizes]


def _rr(case):
    return list(range(1, case["K"] + 1))


def _ints(text):
    return tuple(int(v) for v in text.split(","))


# ---------------------------------------------------------------- inputs
def _chaotic(kind, lengths, rng):
    """FP64 orbits of the given lengths, put together from pieces of SEG samples that are
    iterated side by side (Lorenz: RK4, dt = 0.01, every fifth step, z-scored)."""
    pieces = [-(-n // SEG) for n in lengths]
    p = sum(pieces)
    steps = min(SEG, max(lengths))
    out = np.empty((p, steps))
    if kind == "logistic":
        x = rng.uniform(0.1, 0.9, p)
        for t in range(50 + steps):
            x = 4.0 * x * (1.0 - x)
            x = np.where((x <= 0.0) | (x >= 1.0), 0.3, x)
            if t >= 50:
                out[:, t - 50] = x
    else:
        u = rng.standard_normal((3, p)) * 3.0 + np.array([[1.0], [1.0], [25.0]])

        def f(v):
            return np.stack((10.0 * (v[1] - v[0]), v[0] * (28.0 - v[2]) - v[1], v[0] * v[1] - 8.0 / 3.0 * v[2]))

        h = 0.01
        for t in range(300 + 5 * steps):
            a = f(u)
            b = f(u + 0.5 * h * a)
            c = f(u + 0.5 * h * b)
            d = f(u + h * c)
            u = u + h / 6.0 * (a + 2.0 * b + 2.0 * c + d)
            if t >= 300 and (t - 300) % 5 == 4:
                out[:, (t - 300) // 5] = u[0]
    got, at = [], 0
    for n, k in zip(lengths, pieces):
        x = out[at:at + k].reshape(-1)[:n]
        at += k
        got.append((x - x.mean()) / max(x.std(), 1e-12) if kind == "lorenz" else x)
    return got


def _series(case, seed):
    rng = np.random.default_rng([int(seed) & 0x7FFFFFFF, 17])
    sizes = _sizes(case)
    kinds = [case["signals"] if case["signals"] != "mix" else KINDS[i % 3] for i in range(len(sizes))]
    clean = [None] * len(sizes)
    for kind in ("logistic", "lorenz"):
        at = [i for i, k in enumerate(kinds) if k == kind]
        if at:
            for i, x in zip(at, _chaotic(kind, [sizes[i] for i in at], rng)):
                clean[i] = x
    out = []
    for i, n in enumerate(sizes):
        if clean[i] is None:
            clean[i] = np.sin(2.0 * math.pi * np.arange(n) / 20.3 + rng.uniform(0.0, 2.0 * math.pi))
        snr = SNRS[(i // 3) % 8] if len(sizes) > 4 else (10.0, 0.0, 20.0, -10.0)[i]
        sd = math.sqrt(max(float(np.var(clean[i])), 1e-12) / 10.0 ** (snr / 10.0))
        out.append((clean[i] + sd * rng.standard_normal(n)).astype(np.float32))
    return out


def _given_eps(ys, ms, taus, K, rng):
    """Thresholds a caller brings along: fixed fractions of each series' spread."""
    rows = []
    for y, m, tau in zip(ys, ms, taus):
        ne = len(y) - (m - 1) * tau
        i, j = rng.integers(0, ne, 4000), rng.integers(0, ne, 4000)
        d = np.max([np.abs(y[i + q * tau] - y[j + q * tau]) for q in range(m)], axis=0)
        rows.append(np.quantile(d[i != j], [0.2 * (k + 1) / K for k in range(K)]))
    return np.sort(np.asarray(rows, dtype=np.float32), axis=1)


_STREAMS = []


def _stream():
    """The program's own stream."""
    if not _STREAMS:
        _STREAMS.append(torch.cuda.Stream())
    return _STREAMS[0]


def _net_params(rng):
    parts = []
    for i, o in bracket.LAYERS:
        lim = math.sqrt(6.0 / i)
        parts += [rng.uniform(-lim, lim, o * i), 0.1 * rng.standard_normal(o)]
    return np.concatenate(parts).astype(np.float32)


def prepare(case, seed):
    st = {"case": case}
    what = case["what"]
    if what == "train":
        rng = np.random.default_rng([int(seed) & 0x7FFFFFFF, 23])
        n = 4 * case["rows"]
        feats = np.concatenate([np.sort(rng.normal(0.0, 0.8, (n, 128)), axis=1), rng.uniform(2.0, 4.0, (n, 1)),
                                np.full((n, 2), 3.0)], axis=1)
        labels = np.sort(rng.normal(-1.2, 0.5, (n, 20)), axis=1)
        st["ctx"] = rqa.Context()
        st["X"] = torch.from_numpy(feats.astype(np.float32)).cuda()
        st["T"] = torch.from_numpy(labels.astype(np.float32)).cuda()
        st["idx"] = torch.from_numpy(rng.permutation(n)[:case["rows"]].astype(np.int64)).cuda()
        st["params0"] = torch.from_numpy(_net_params(rng)).cuda()
        B = case["rows"]
        for name, shape in (("xb", (B, 131)), ("tb", (B, 20)), ("Y", (B, 40)), ("acts", (B, rqa.RQA_MLP_ACTS)),
                            ("loss", (1,)), ("grads", (rqa.RQA_MLP_PARAMS,)), ("m", (rqa.RQA_MLP_PARAMS,)),
                            ("v", (rqa.RQA_MLP_PARAMS,))):
            st[name] = torch.zeros(shape, dtype=torch.float32, device="cuda")
        return st
    ys = _series(case, seed)
    ms, taus = _embedding(case, [len(y) for y in ys])
    st["batch"] = rqa.Batch.from_numpy(ys, ms, taus)
    if what in ("lines", "vlines"):
        rng = np.random.default_rng([int(seed) & 0x7FFFFFFF, 29])
        st["eps"] = torch.from_numpy(_given_eps(ys, ms, taus, case["K"], rng)).cuda()
    if what == "det" and case["kept"]:
        # a program that calls again and again: its own stream and its own output buffers
        S, K, lmin = len(ys), case["K"], _ints(case["lmin"])
        torch.cuda.synchronize()
        st["ctx"] = rqa.Context(stream=_stream())
        if case["learned"]:
            bracket.install(st["ctx"])
        st["hoff"] = st["batch"].hist_offsets(K)
        f64 = {"dtype": torch.float64, "device": "cuda"}
        st["det"] = torch.empty((S, K, len(lmin)), **f64)
        st["avg"] = torch.empty((S, len(lmin)), **f64)
        st["eps"] = torch.empty((S, K), dtype=torch.float32, device="cuda")
        st["hist"] = torch.empty(int(st["hoff"][-1]), dtype=torch.uint64, device="cuda") if case["lines"] else None
        st["lmax"] = torch.empty((S, K), dtype=torch.uint32, device="cuda")
        st["count"] = torch.empty((S, K), dtype=torch.uint64, device="cuda")
        st["stencil"] = torch.empty((S, K), dtype=torch.uint64, device="cuda")
    elif what == "labels":
        S = len(ys)
        st["ctx"] = rqa.Context(select=rqa.RQA_SELECT_RADIX)
        st["eps"] = torch.empty((S, 20), dtype=torch.float32, device="cuda")
        st["X"] = torch.empty((S, 131), dtype=torch.float32, device="cuda")
        st["centre"] = torch.empty(S, dtype=torch.float32, device="cuda")
        st["T"] = torch.empty((S, 20), dtype=torch.float32, device="cuda")
    elif what == "noalloc":
        S, K = len(ys), case["K"]
        st["eps"] = torch.empty((S, K), dtype=torch.float32, device="cuda")
        st["le"] = torch.empty((S, K), dtype=torch.uint64, device="cuda")
        st["lt"] = torch.empty((S, K), dtype=torch.uint64, device="cuda")
        st["status"] = torch.empty(1, dtype=torch.int32, device="cuda")
    else:
        st["ctx"] = rqa.Context()
        if what == "det" and case["learned"]:
            bracket.install(st["ctx"])
    return st


# ---------------------------------------------------------------- one pass
def _signed(out):
    """Counts as int64 views: torch indexes those."""
    return {k: v.view(torch.int64) if v.dtype == torch.uint64 else v for k, v in out.items()}


def run(st):
    case = st["case"]
    what = case["what"]
    if what == "det":
        rr, lmin = _rr(case), _ints(case["lmin"])
        if not case["kept"]:
            out = rqa.det_avg(st["ctx"], st["batch"], rr, case["den"], lmin=lmin, lines=case["lines"])
            out.pop("hist_offsets", None)
            return _signed(out)
        hoff = st["hoff"] if case["lines"] else None
        rqa.rqa_det_avg(st["ctx"], st["batch"], rr, case["den"], None, case["K"], lmin, st["det"], st["avg"],
                        st["eps"], st["hist"], hoff, st["lmax"], st["count"], st["stencil"])
        return _signed({k: st[k] for k in ("det", "avg", "eps", "hist", "lmax", "count", "stencil")
                        if st[k] is not None})
    if what == "eps":
        return rqa.eps_for_rr(st["ctx"], st["batch"], _rr(case), case["den"])
    if what == "lines":
        lh = rqa.line_hist(st["ctx"], st["batch"], st["eps"], case["K"])
        lm = rqa.line_measures(st["ctx"], st["batch"], lh["hist"], lh["hist_offsets"], case["K"], _ints(case["lmin"]))
        lh.pop("hist_offsets")
        return _signed({**lh, **lm})
    if what == "vlines":
        vh = rqa.vline_hist(st["ctx"], st["batch"], st["eps"], case["K"])
        lt = rqa.lam_tt(st["ctx"], st["batch"], vh["vhist"], vh["vhist_offsets"], case["K"], _ints(case["vmin"]))
        vh.pop("vhist_offsets")
        return _signed({**vh, **lt})
    if what == "grid":
        g = rqa.eps_approx(st["ctx"], st["batch"], _rr(case), case["den"], case["n_thr"])
        d = rqa.det_avg(st["ctx"], st["batch"], None, 0, eps=g["eps"], K=case["K"])
        return {**g, "det": d["det"], "det_avg": d["det_avg"]}
    if what == "train":
        ctx = st["ctx"]
        params = st["params0"].clone()  # every pass is the first step from the same weights
        st["m"].zero_()
        st["v"].zero_()
        rqa.rqa_gather_rows(ctx, st["X"], st["idx"], st["xb"])
        rqa.rqa_gather_rows(ctx, st["T"], st["idx"], st["tb"])
        rqa.rqa_mlp_forward(ctx, params, st["xb"], st["Y"], st["acts"])
        rqa.rqa_mlp_backward(ctx, params, st["xb"], st["acts"], st["Y"], st["tb"], 0.005, 0.995, st["grads"],
                             st["loss"])
        rqa.rqa_adam_step(ctx, params, st["grads"], st["m"], st["v"], 1, 2e-3)
        return {"Y": st["Y"], "loss": st["loss"], "grads": st["grads"], "m": st["m"], "v": st["v"]}
    if what == "labels":
        ctx, b = st["ctx"], st["batch"]
        rqa.rqa_eps_for_rr(ctx, b, bracket.RR, 100, st["eps"])
        rqa.rqa_sketch(ctx, b, 1, st["X"], st["centre"])
        rqa.rqa_log_labels(ctx, st["eps"], st["centre"], st["T"])
        return {k: st[k] for k in ("eps", "X", "centre", "T")}
    rqa.rqa_eps_for_rr_noalloc(st["batch"], _rr(case), case["den"], st["eps"], st["le"], st["lt"], st["status"])
    return {k: st[k] for k in ("eps", "le", "lt", "status")}


# ---------------------------------------------------------------- work
def work(case):
    """Inputs read once, outputs written once; one distance (2 m - 1 operations) per cell for the
    selection and one for the line pass, which needs the thresholds first."""
    what = case["what"]
    if what == "train":
        B, P = case["rows"], sum(i * o for i, o in bracket.LAYERS)
        n = rqa.RQA_MLP_PARAMS
        return {"bytes": 4 * (B * (131 + 20 + 40) + 8 * n), "flops": 2 * B * P * 3 - 2 * B * 131 * 256 + 12 * n}
    sizes = _sizes(case)
    ms, taus = _embedding(case, sizes)
    passes = {"det": 2, "eps": 1, "lines": 1, "vlines": 2, "grid": 2, "labels": 1, "noalloc": 1}[what]
    flops, rows = 0, 0
    for n, m, tau in zip(sizes, ms, taus):
        ne = n - (m - 1) * tau
        flops += passes * (2 * m - 1) * ne * (ne - 1) // 2
        rows += ne - 1
    S, K = len(sizes), case.get("K", 20)
    out = S * K * 28
    if what in ("lines", "vlines") or case.get("lines"):
        out += 8 * K * rows
    if what == "labels":
        out += S * 4 * 152
    return {"bytes": 4 * sum(sizes) + out, "flops": flops}


# ---------------------------------------------------------------- exact values
def _matrix(y, m, tau):
    """FP32 maximum-norm distances (the definition's own type) of all pairs, on the GPU."""
    y = torch.from_numpy(y).cuda()
    ne = y.numel() - (m - 1) * tau
    d = torch.zeros((ne, ne), dtype=torch.float32, device="cuda")
    for q in range(m):
        x = y[q * tau:q * tau + ne]
        torch.maximum(d, (x[:, None] - x[None, :]).abs(), out=d)
    return d


def _diagonals(d):
    """Row s = the diagonal j - i = s + 1 of d, padded by inf to one length."""
    ne = d.shape[0]
    i = torch.arange(ne, device=d.device)[None, :]
    j = i + torch.arange(1, ne, device=d.device)[:, None]
    x = d[i.expand(ne - 1, ne), j.clamp(max=ne - 1)]
    return torch.where(j < ne, x, torch.full_like(x, math.inf))


def _runs(rec):
    """Histogram over lengths 0.. of the runs of True along the rows."""
    flat = torch.nn.functional.pad(rec.to(torch.int8), (1, 1)).reshape(-1)
    step = flat[1:] - flat[:-1]
    start = torch.nonzero(step == 1).reshape(-1)
    end = torch.nonzero(step == -1).reshape(-1)
    return torch.bincount(end - start, minlength=rec.shape[1] + 1)


def _measures(hist, lmin):
    l = torch.arange(hist.numel(), dtype=torch.int64, device=hist.device)
    return [(int((hist * l)[a:].sum()), int(hist[a:].sum()), hist[a:]) for a in lmin]


def _ratio(a, b):
    return a / b if b else math.nan


def _exact_lines(rec_of, eps, lmin):
    """DET or LAM, L or TT and ENTR per threshold and minimal length."""
    det, L, ent = [], [], []
    for e in eps:
        h = _runs(rec_of(e))
        total = _measures(h, (1,))[0][0]
        ms = _measures(h, lmin)
        det.append([_ratio(a, total) for a, _, _ in ms])
        L.append([_ratio(a, n) for a, n, _ in ms])
        row = []
        for _, n, part in ms:
            p = part[part > 0].double() / max(n, 1)
            row.append(float(-(p * p.log()).sum()) if n else 0.0)
        ent.append(row)
    return tuple(torch.tensor(v, dtype=torch.float64) for v in (det, L, ent))


def _exact_eps(d, K, den):
    ne = d.shape[0]
    i = torch.triu_indices(ne, ne, 1, device=d.device)
    v, _ = torch.sort(d[i[0], i[1]])
    P = v.numel()
    return [float(v[-(-k * P // den) - 1]) for k in range(1, K + 1)], v


def exact(case, seed):
    what = case["what"]
    if what == "train":
        st = prepare(case, seed)
        p = st["params0"].double().requires_grad_(True)
        x, t = st["X"][st["idx"]].double(), st["T"][st["idx"]].double()
        at, h = 0, x
        for k, (i, o) in enumerate(bracket.LAYERS):
            w, b = p[at:at + o * i].reshape(o, i), p[at + o * i:at + o * i + o]
            at += o * i + o
            h = h @ w.T + b
            h = h.relu() if k < 2 else h
        tau = torch.tensor([0.005, 0.995], dtype=torch.float64, device="cuda").repeat(20)
        r = t.repeat_interleave(2, dim=1) - h
        loss = torch.where(r >= 0, tau * r, (tau - 1.0) * r).mean()
        loss.backward()
        g = p.grad
        return {"Y": h.detach(), "loss": loss.detach().reshape(1), "grads": g, "m": 0.1 * g, "v": 0.001 * g * g}
    sizes = _sizes(case)
    if what == "labels" or sum(n * n for n in sizes) * case.get("K", 20) > 1.2e10 or max(sizes) > 10000:
        return None
    ys = _series(case, seed)
    ms, taus = _embedding(case, sizes)
    K = case["K"]
    given = None
    if what in ("lines", "vlines"):
        rng = np.random.default_rng([int(seed) & 0x7FFFFFFF, 29])
        given = _given_eps(ys, ms, taus, K, rng)
    if what == "vlines":
        lmin = _ints(case["vmin"])
    else:
        lmin = _ints(case.get("lmin", "2"))
    eps_all, det_all, l_all, e_all, rr_all = [], [], [], [], []
    for s, (y, m, tau) in enumerate(zip(ys, ms, taus)):
        d = _matrix(y, m, tau)
        ne = d.shape[0]
        if given is not None:
            eps = [float(v) for v in given[s]]
        elif what == "grid":
            n = case["n_thr"]
            scale = np.float32(np.float32(y.max() - y.min()) / np.float32(n))
            grid = (np.arange(1, n + 1, dtype=np.float32) * scale).astype(np.float32)
            i = torch.triu_indices(ne, ne, 1, device=d.device)
            v, _ = torch.sort(d[i[0], i[1]])
            c = torch.searchsorted(v, torch.from_numpy(grid).cuda(), right=True).cpu().numpy().astype(object)
            P = v.numel()
            best = [min(range(n), key=lambda j: (abs(c[j] * case["den"] - k * P), j)) for k in range(1, K + 1)]
            eps = [float(grid[b]) for b in best]
            rr_all.append([float(int(c[b]) / P) for b in best])
        else:
            eps, _ = _exact_eps(d, K, case["den"])
        eps_all.append(eps)
        if what in ("det", "lines", "grid"):
            x = _diagonals(d)
            a = _exact_lines(lambda e: x <= e, eps, lmin)
        elif what == "vlines":
            x = d.clone()
            x.fill_diagonal_(math.inf)
            x = x.T.contiguous()
            a = _exact_lines(lambda e: x <= e, eps, lmin)
        else:
            continue
        det_all.append(a[0])
        l_all.append(a[1])
        e_all.append(a[2])
    eps = torch.tensor(eps_all, dtype=torch.float64)
    if what == "eps":
        return {"eps": eps, "count_le": None, "count_lt": None}
    if what == "noalloc":
        return {"eps": eps, "le": None, "lt": None, "status": None}
    det = torch.stack(det_all)
    if what == "det":
        return {"det": det, "avg" if case["kept"] else "det_avg": det.mean(dim=1), "eps": eps}
    if what == "grid":
        return {"eps": eps, "rr": torch.tensor(rr_all, dtype=torch.float64), "count": None, "det": det,
                "det_avg": det.mean(dim=1)}
    L, E = torch.stack(l_all), torch.stack(e_all)
    if what == "vlines":
        return {"lam": det, "tt": L, "lam_avg": det.mean(dim=1), "tt_avg": L.mean(dim=1)}
    return {"L": L, "entr": E, "L_avg": L.mean(dim=1), "entr_avg": E.mean(dim=1)}
