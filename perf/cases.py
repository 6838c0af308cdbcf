"""The calls whose speed this framework is measured by, through its public
binding (``paper_2404_12134_gb300.api``), with inputs made on the GPU from a
seed.

Each case names the work it stands for.  The sizes are those of the five
workloads of ``synth.py``, of the segmentation setting and of the small batches
of the tests; ``draw`` gives further cases over the same ranges.  Signals
follow the recipe of ``synth.py`` (smooth quasi-periodic channels, a monotone
piecewise-linear time warp per cycle, noise, removed gaps, some anomalous
cycles), drawn with torch on the GPU.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2404_12134_gb300 import api


def listed():
    return [
        # one new cycle scored as it arrives: the smallest call, bound by latency and launches
        {"name": "score_one", "op": "score", "T": 1, "lo": 1100, "hi": 1100, "M": 1087, "d": 1},
        # one averaging iteration over a small set of short cycles (the smallest workload)
        {"name": "dba_small", "op": "dba", "T": 16, "lo": 1000, "hi": 1200, "M": 1093, "d": 1},
        # one averaging iteration of the benchmark batch: long six-channel cycles
        {"name": "dba_batch", "op": "dba", "T": 200, "lo": 20000, "hi": 30000, "M": 25000, "d": 6},
        # a fleet of very uneven cycles scored against a fixed prototype
        {"name": "score_uneven", "op": "score", "T": 1000, "lo": 2000, "hi": 60000, "M": 20000, "d": 3},
        # alignment paths under the l2 norm itself (Sec. 3.2's wording), a handful of cycles
        {"name": "align_l2", "op": "align", "T": 24, "lo": 7000, "hi": 9500, "M": 8191, "d": 6, "l2": True},
        # the averaging loop's start: pairwise costs of 16 cycles, their medoid, resampled
        {"name": "medoid_init", "op": "medoid", "T": 16, "lo": 20000, "hi": 30000, "M": 25000, "d": 6},
        # a training step of the Soft-DTW barycenter: values and gradient through autograd
        {"name": "soft_train", "op": "soft", "T": 64, "lo": 8000, "hi": 12000, "M": 10000, "d": 1, "gamma": 0.1},
        # the same with several channels and few, short cycles
        {"name": "soft_small", "op": "soft", "T": 16, "lo": 900, "hi": 1300, "M": 1111, "d": 6, "gamma": 1.0},
        # Table I's setting: gamma 1, Sakoe-Chiba band 0.6
        {"name": "soft_band", "op": "soft", "T": 64, "lo": 8000, "hi": 12000, "M": 10000, "d": 1, "gamma": 1.0,
         "band": 0.6},
        # cycles too long to keep R: column checkpoints, R recomputed in the backward
        {"name": "soft_long", "op": "soft", "T": 8, "lo": 100000, "hi": 120000, "M": 110000, "d": 3, "gamma": 0.1,
         "ckpt": True},
        # averaging over very long cycles with the codes recomputed from checkpoints
        {"name": "dba_long", "op": "dba", "T": 32, "lo": 100000, "hi": 120000, "M": 110000, "d": 3, "ckpt": True},
        # a day's stream cut into cycles by Sub-DTW windows against a reference cycle
        {"name": "segment", "op": "segment", "T": 36, "lo": 15000, "hi": 18000, "M": 16283, "d": 9},
    ]


def _log(rng, a, b):
    return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))


def draw(rng):
    op = rng.choice(["score", "score", "dba", "dba", "align", "medoid", "soft", "soft", "soft", "segment"])
    c = {"op": op}
    if op == "segment":
        M = _log(rng, 900, 16300)
        c.update(T=_log(rng, 4, 30), lo=int(0.92 * M) | 1, hi=int(1.1 * M), M=M, d=rng.choice([1, 3, 6, 9]))
        return c
    if op == "soft":
        # up to the cells of soft_train with R kept, of a tenth of soft_long with checkpoints
        ckpt = rng.random() < 0.3
        cells = math.exp(rng.uniform(math.log(1.5e7), math.log(9e9 if ckpt else 5e9)))
        M = _log(rng, 900, 40000 if ckpt else 12000)
        T = max(1, min(64, int(cells / (M * 1.1 * M))))
        c.update(T=T, lo=int(0.75 * M) | 1, hi=int(1.25 * M), M=M, d=rng.choice([1, 1, 2, 3, 6, 8]),
                 gamma=rng.choice([1.0, 0.1, 0.01]))
        if ckpt:
            c["ckpt"] = True
        elif rng.random() < 0.35:
            c["band"] = rng.choice([0.3, 0.6])
        return c
    cells = math.exp(rng.uniform(math.log(1e6), math.log(1.0e11)))
    if op == "medoid":
        M = _log(rng, 900, 25000)
        T = max(3, min(16, int(math.sqrt(2 * min(cells, 5e10) / (M * M)))))
        c.update(T=T, lo=int(0.8 * M) | 1, hi=int(1.2 * M), M=M, d=rng.choice([1, 2, 3, 6, 9]))
        return c
    M = _log(rng, 900, 30000)
    T = max(1, min(400, int(cells / (M * M))))
    d = rng.choice([1, 1, 2, 3, 3, 4, 6, 6, 9, 12])
    wide = op == "score" and rng.random() < 0.5
    c.update(T=T, lo=max(500, int((0.3 if wide else 0.8) * M)) | 1, hi=max(1000, int((1.7 if wide else 1.2) * M)), M=M,
             d=d)
    if op == "align":
        if rng.random() < 0.4:
            c["l2"] = True
        elif rng.random() < 0.4:
            c["band"] = rng.choice([0.1, 0.3, 0.6])
    if op == "dba" and rng.random() < 0.25:
        c["ckpt"] = True
    return c


# --- inputs --------------------------------------------------------------------

def _rand(g, *size, lo=0.0, hi=1.0):
    return torch.rand(*size, generator=g, device="cuda") * (hi - lo) + lo


class _Signal:
    """A smooth z-normalised function of t in [0, 1) with d channels: Gaussian
    bumps and sinusoids (five sinusoids for a single channel)."""

    def __init__(self, g, d):
        nb, ns = (0, 5) if d == 1 else (8, 2)
        self.centre = _rand(g, nb, d)
        self.width = _rand(g, nb, d, lo=0.01, hi=0.08)
        self.bump = torch.randn(nb, d, generator=g, device="cuda")
        self.period = _rand(g, ns, d, lo=50.0, hi=400.0) / 1100.0
        self.amp = _rand(g, ns, d, lo=0.2, hi=1.0)
        self.phase = _rand(g, ns, d, hi=2 * math.pi)
        self.mu, self.sd = 0.0, 1.0
        grid = self((torch.arange(4096, device="cuda") + 0.5) / 4096)
        self.mu, self.sd = grid.mean(0), grid.std(0)

    def __call__(self, t):
        t = t[:, None]
        out = torch.zeros((), device="cuda")
        for k in range(self.amp.shape[0]):
            out = out + self.amp[k] * torch.sin(2 * math.pi * t / self.period[k] + self.phase[k])
        for k in range(self.bump.shape[0]):
            out = out + self.bump[k] * torch.exp(-0.5 * ((t - self.centre[k]) / self.width[k]) ** 2)
        return (out - self.mu) / self.sd


def _cycles(g, signal, lengths, noise=0.05):
    """Warped, noisy cycles of the signal with gaps removed, packed: (data, offsets)."""
    T = len(lengths)
    L = torch.tensor(lengths, device="cuda")
    start = torch.cumsum(L, 0) - L
    cyc = torch.repeat_interleave(torch.arange(T, device="cuda"), L)
    n = int(cyc.numel())
    x = (torch.arange(n, device="cuda") - start[cyc]).float() / L[cyc].float()
    knots = torch.sort(_rand(g, T, 8), dim=1).values
    knots = torch.cat([torch.zeros(T, 1, device="cuda"), knots, torch.ones(T, 1, device="cuda")], 1)
    slope = _rand(g, T, 9, lo=0.7, hi=1.4)
    total = (slope * (knots[:, 1:] - knots[:, :-1])).sum(1)
    u = torch.zeros(n, device="cuda")
    for k in range(9):
        a, b = knots[:, k][cyc], knots[:, k + 1][cyc]
        u += slope[:, k][cyc] * torch.minimum(x - a, b - a).clamp_(min=0)
    u /= total[cyc]
    # one cycle in ten is anomalous: it drifts, or skips 5 % of the signal
    kind = torch.where(_rand(g, T) < 0.1, torch.where(_rand(g, T) < 0.5, 1, 2), 0)
    at = _rand(g, T, hi=0.7)
    u = torch.where(kind[cyc] == 2, torch.where(0.95 * u < at[cyc], 0.95 * u, 0.95 * u + 0.05), u)
    y = signal(u)
    ramp = ((x - at[cyc]) / 0.3).clamp_(0.0, 1.0) * 0.5
    y += torch.where(kind[cyc] == 1, ramp, torch.zeros((), device="cuda"))[:, None]
    y += noise * torch.randn(y.shape, generator=g, device="cuda")
    # 2 % of the time steps missing, in runs of 5 to 20 (a cycle's first step stays)
    run = torch.randint(5, 21, (n,), generator=g, device="cuda")
    starts = torch.nonzero(_rand(g, n) < 0.02 / 12.5).flatten()
    edge = torch.zeros(n + 32, dtype=torch.int32, device="cuda")
    one = torch.ones(starts.numel(), dtype=torch.int32, device="cuda")
    edge.index_add_(0, starts, one)
    edge.index_add_(0, starts + run[starts], -one)
    keep = torch.cumsum(edge, 0)[:n] <= 0
    keep[start] = True
    offsets = torch.zeros(T + 1, dtype=torch.int64, device="cuda")
    offsets[1:] = torch.cumsum(torch.zeros(T, dtype=torch.int64, device="cuda").index_add_(0, cyc, keep.long()), 0)
    return y[keep].contiguous(), offsets


def _inputs(case, seed):
    """(signal, batch data, offsets, prototype) of a case."""
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    r = np.random.default_rng(int(seed))
    T, lo, hi = case["T"], case["lo"], case["hi"]
    if hi > 8 * lo:                 # very uneven: log-normal, as the scoring workload's
        lengths = np.clip(np.exp(r.normal(0.5 * math.log(lo * hi) + 0.3, 0.6, T)), lo, hi).astype(int)
    else:
        lengths = r.integers(lo, hi + 1, T)
    signal = _Signal(g, case["d"])
    data, offsets = _cycles(g, signal, lengths.tolist())
    M = case["M"]
    B = signal((torch.arange(M, device="cuda") + 0.5) / M)
    if case["op"] in ("dba", "soft", "segment"):
        # a prototype in the making (or an operator's pick) still carries some noise
        B = B + 0.03 * torch.randn(B.shape, generator=g, device="cuda")
    return data, offsets, B.float().contiguous()


def _options(case):
    return api.options(band=case.get("band", 0.0), cost_kind=1 if case.get("l2") else 0,
                       dir_mode=1 if case.get("ckpt") else 0)


class _State:
    pass


def prepare(case, seed):
    s = _State()
    s.case = case
    data, offsets, s.B = _inputs(case, seed)
    s.opts = _options(case)
    s.ws = api.Workspace()
    if case["op"] == "segment":
        s.Y = data
        return s
    s.batch = api.Batch(data, offsets)
    if case["op"] == "soft":
        s.w = torch.from_numpy((1.0 / s.batch.lengths).astype(np.float32)).cuda()
        s.B.requires_grad_(True)
    return s


def run(s):
    op = s.case["op"]
    if op == "score":
        score, cost, plen = api.anomaly_score(s.B, s.batch, s.opts, s.ws)
        return {"score": score, "cost": cost, "plen": plen}
    if op == "dba":
        B, counts, before, cost = api.dba_iterate(s.B, s.batch, s.opts, s.ws)
        return {"B": B, "counts": counts, "before": before, "cost": cost}
    if op == "align":
        cost, plen, jlo, jhi = api.dtw_align(s.B, s.batch, s.opts, s.ws)
        return {"cost": cost, "plen": plen, "jlo": jlo, "jhi": jhi}
    if op == "medoid":
        C = api.pairwise_dtw(s.batch, s.opts, s.ws)
        index, sums = api.medoid(C)
        k = int(index)
        o = s.batch.offsets_host
        return {"C": C, "index": index, "sums": sums, "B": api.resample(s.batch.data[o[k]:o[k + 1]], s.case["M"])}
    if op == "soft":
        values = api.softdtw(s.B, s.batch, s.case["gamma"], s.opts)
        grad, = torch.autograd.grad(values, s.B, s.w)
        return {"values": values.detach(), "grad": grad}
    found = api.segment(s.B, s.Y, opts=s.opts, ws=s.ws)
    # the pieces in a table with room for more, so that its shape does not hang on the stream
    bounds = np.full((4 * s.case["T"] + 64, 2), -1, dtype=np.int64)
    cost = np.zeros(bounds.shape[0], dtype=np.float32)
    for k, (first, last, c) in enumerate(found):
        bounds[k] = first, last
        cost[k] = c
    return {"count": len(found), "bounds": bounds, "cost": cost}


def work(case):
    """Inputs read once, outputs written once; 2 d operations a cell for the
    local cost and 3 for the recursion (Soft-DTW: about 14 forward, and 2 d + 16
    backward)."""
    T, M, d, op = case["T"], case["M"], case["d"], case["op"]
    n = math.exp(0.5 * math.log(case["lo"] * case["hi"]) + 0.48) if case["hi"] > 8 * case["lo"] else 0.5 * (
        case["lo"] + case["hi"])
    n *= 0.98
    cells = T * M * n
    data = 4.0 * d * (T * n + M)
    cell_ops = 2 * d + 3 + (1 if case.get("l2") else 0)
    if case.get("band"):
        w = min(1.0, case["band"])
        cells *= 1 - (1 - w) ** 2
    if op == "score":
        return {"bytes": data + 12 * T, "flops": cells * cell_ops}
    if op == "dba":
        return {"bytes": data + 4 * M * (d + 1) + 4 * T, "flops": cells * cell_ops}
    if op == "align":
        return {"bytes": data + 8 * T * M, "flops": cells * cell_ops}
    if op == "medoid":
        return {"bytes": data + 4 * T * T + 4 * M * d, "flops": 0.5 * T * (T - 1) * n * n * cell_ops}
    if op == "soft":
        return {"bytes": data + 4 * T + 4 * M * d, "flops": cells * (2 * d + 14 + 2 * d + 16)}
    # windows of 2 M, one a cycle
    return {"bytes": data + 16 * T, "flops": T * 2.0 * M * M * cell_ops}


# --- the same in 64 bits ----------------------------------------------------------

class _Diagonals:
    """The anti-diagonals of all T matrices at once: the local costs of
    diagonal s for rows 0 .. M-1 (inf outside a matrix)."""

    def __init__(self, case, data, offsets, B):
        self.o = offsets.cpu().numpy()
        self.N = torch.from_numpy(np.diff(self.o)).cuda()
        self.T, self.M, self.d = case["T"], B.shape[0], B.shape[1]
        self.n = int(self.N.max())
        self.B = B.detach().double()
        # reversed cycles, inf around them: diagonal s is a contiguous slice over the rows
        self.Y = torch.full((self.T, self.n + 2 * self.M, self.d), math.inf, dtype=torch.float64, device="cuda")
        for k in range(self.T):
            y = data[int(self.o[k]):int(self.o[k + 1])].double().flip(0)
            at = self.M + self.n - y.shape[0]
            self.Y[k, at:at + y.shape[0]] = y
        self.count = self.M + self.n - 1
        self.l2 = bool(case.get("l2"))
        self.inf = torch.full((self.T, 1), math.inf, dtype=torch.float64, device="cuda")

    def y(self, s):
        at = self.M + self.n - 1 - s
        return self.Y[:, at:at + self.M]

    def cost(self, s):
        c = ((self.B - self.y(s)) ** 2).sum(2)
        return c.sqrt() if self.l2 else c

    def last(self, history):
        """The last cell of every matrix from row M - 1 of each diagonal."""
        return history[self.N + self.M - 2, torch.arange(self.T, device="cuda")]


def _dtw64(diag, codes=False):
    """Costs [T], and every cell's code (0 diagonal, 1 up, 2 left) by diagonal."""
    T, M = diag.T, diag.M
    p1 = torch.full((T, M + 1), math.inf, dtype=torch.float64, device="cuda")
    p2 = p1.clone()
    p2[:, 0] = 0.0
    history = torch.empty(diag.count, T, dtype=torch.float64, device="cuda")
    kept = torch.empty(diag.count, T, M, dtype=torch.uint8, device="cuda") if codes else None
    for s in range(diag.count):
        dg, up, lf = p2[:, :-1], p1[:, :-1], p1[:, 1:]
        m = torch.minimum(torch.minimum(dg, up), lf)
        if codes:
            kept[s] = torch.where(dg == m, 0, torch.where(up == m, 1, 2)).to(torch.uint8)
        r = torch.cat([diag.inf, diag.cost(s) + m], 1)
        history[s] = r[:, M]
        p2, p1 = p1, r
    return diag.last(history), kept


def _dba64(diag, data):
    cost, kept = _dtw64(diag, codes=True)
    kept, N = kept.cpu().numpy(), diag.N.cpu().numpy()
    total = np.zeros((diag.M, diag.d))
    count = np.zeros(diag.M)
    y = data.double().cpu().numpy()
    for k in range(diag.T):
        i, j = diag.M - 1, int(N[k]) - 1
        while True:
            total[i] += y[diag.o[k] + j]
            count[i] += 1
            if i == 0 and j == 0:
                break
            c = kept[i + j, k, i]
            i, j = i - (c != 2), j - (c != 1)
    return total / count[:, None], cost


def _soft64(diag, gamma, weights=None):
    """Values [T] and, with weights, the gradient [M, d]."""
    T, M = diag.T, diag.M
    p1 = torch.full((T, M + 1), math.inf, dtype=torch.float64, device="cuda")
    p2 = p1.clone()
    p2[:, 0] = 0.0
    history = torch.empty(diag.count, T, dtype=torch.float64, device="cuda")
    R = torch.empty(diag.count, T, M, dtype=torch.float64, device="cuda") if weights is not None else None
    for s in range(diag.count):
        m = -gamma * torch.logsumexp(torch.stack([p2[:, :-1], p1[:, :-1], p1[:, 1:]]) / -gamma, 0)
        r = torch.cat([diag.inf, diag.cost(s) + m], 1)
        history[s] = r[:, M]
        if R is not None:
            R[s] = r[:, 1:]
        p2, p1 = p1, r
    values = diag.last(history)
    if weights is None:
        return values, None
    zero = torch.zeros(T, M + 1, dtype=torch.float64, device="cuda")
    e1, e2 = zero.clone(), zero.clone()                     # diagonals s + 1, s + 2 (row M: beyond the matrix)
    v1 = torch.full((T, M + 1), -math.inf, dtype=torch.float64, device="cuda")   # r - delta there
    v2 = v1.clone()
    grad = torch.zeros(M, diag.d, dtype=torch.float64, device="cuda")
    row = torch.arange(M, device="cuda")
    for s in range(diag.count - 1, -1, -1):
        r = R[s]
        inside = torch.isfinite(r)
        rs = torch.where(inside, r, torch.zeros((), dtype=torch.float64, device="cuda"))
        e = sum(torch.exp((v - rs) / gamma) * x for v, x in ((v1[:, 1:], e1[:, 1:]), (v1[:, :-1], e1[:, :-1]),
                                                             (v2[:, 1:], e2[:, 1:])))
        e = torch.where((row == M - 1) & (diag.N[:, None] - 1 == s - row), torch.ones_like(e), e)
        e = torch.where(inside, e, torch.zeros_like(e))
        t = torch.where(inside[:, :, None], diag.B - diag.y(s), torch.zeros((), dtype=torch.float64, device="cuda"))
        grad += 2.0 * ((weights[:, None] * e)[:, :, None] * t).sum(0)
        v = torch.where(inside, r - diag.cost(s), torch.full_like(r, -math.inf))
        e2, v2 = e1, v1
        e1 = torch.cat([e, zero[:, :1]], 1)
        v1 = torch.cat([v, torch.full_like(zero[:, :1], -math.inf)], 1)
    return values, grad


def exact(case, seed):
    op = case["op"]
    if op in ("segment", "medoid") or case.get("band"):
        return None
    n = 0.5 * (case["lo"] + case["hi"]) if case["hi"] <= 8 * case["lo"] else case["hi"]
    diagonals, cells = case["M"] + case["hi"], case["T"] * case["M"] * n
    seconds = diagonals * 2.5e-4 + cells * (2 * case["d"] + 8) * (1e-10 if op == "soft" else 2e-12)
    if seconds > 12:
        return None
    data, offsets, B = _inputs(case, seed)
    diag = _Diagonals(case, data, offsets, B)
    if op == "score":
        return {"score": None, "cost": _dtw64(diag)[0], "plen": None}
    if op == "align":
        return {"cost": _dtw64(diag)[0], "plen": None, "jlo": None, "jhi": None}
    if op == "dba":
        if diagonals * case["T"] * case["M"] > 2e9:
            cost = _dtw64(diag)[0]
            return {"B": None, "counts": None, "before": cost.sum(), "cost": cost}
        mean, cost = _dba64(diag, data)
        return {"B": mean, "counts": None, "before": cost.sum(), "cost": cost}
    small = diagonals * case["T"] * case["M"] * 8 < 4e9
    values, grad = _soft64(diag, case["gamma"], 1.0 / diag.N.double() if small else None)
    return {"values": values, "grad": grad}
