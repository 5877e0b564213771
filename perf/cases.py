"""The work that users of this library have it do, as timed cases.

A read mapper calls the library in a few ways: whole batches of extensions on
the device or from host buffers, a handful of reads at a time, a stream of
requests through the server, and the same with CIGARs or in the local
(BWA-MEM) variant.  The listed cases are the repository's workloads (small,
ONT-like, HiFi-like, skewed, short reads, serving) through those entry points;
`draw` spreads over the same lengths, batch sizes, bands and scorings.

Inputs are random reads and their mutated references, as
`paper_2403_06478_gb300.workload` describes them, drawn on the GPU so that a
hundred million bases take well under a second.
"""
import math

import numpy as np
import torch

from paper_2403_06478_gb300 import agatha as A
from paper_2403_06478_gb300.workload import Scoring

DEV = "cuda" if torch.cuda.is_available() else "cpu"

# error rates (sub, ins, del), divergent-tail fraction of each read technology
ERRORS = {
    "small": (0.05, 0.025, 0.025, 0.0),
    "ont": (0.05, 0.03, 0.04, 0.10),
    "hifi": (0.005, 0.0025, 0.0025, 0.02),
    "skewed": (0.04, 0.02, 0.02, 0.20),
    "short": (0.008, 0.001, 0.001, 0.05),
}
# a, b, q, e, q2, e2, zdrop, end_bonus
SCORES = {
    "ont": (2, 4, 4, 2, 24, 1, 400, 0),
    "hifi": (1, 4, 6, 2, 26, 1, 200, 0),
    "bwa": (1, 4, 6, 1, 6, 1, 100, 5),
}


def listed():
    return [
        # the smallest call: a few short reads from host buffers, all latency
        dict(name="reads16_host", api="host", pairs=16, dist="fixed", length=150, errors="short",
             scores="bwa", w=100, tuned=False),
        # one small batch from host buffers: 256 extensions of 1 kbp
        dict(name="small_host", api="host", pairs=256, dist="fixed", length=1000, errors="small",
             scores="ont", w=100, tuned=False),
        # the benchmark's batch end to end, on an autotuned context as the benchmark runs it
        dict(name="ont_host", api="host", pairs=20000, dist="lognormal", length=5000, errors="ont",
             scores="ont", w=500, tuned=True),
        # accurate long reads already on the device
        dict(name="hifi_device", api="device", pairs=5000, dist="normal", length=15000, errors="hifi",
             scores="hifi", w=500, tuned=False),
        # a Pareto mix of lengths at a wide band, a fifth of them ending in a Z-drop
        dict(name="skewed_device", api="device", pairs=100000, dist="pareto", length=500, errors="skewed",
             scores="ont", w=750, tuned=False),
        # short reads with BWA-MEM's parameters (single-piece gaps)
        dict(name="short_device", api="device", pairs=200000, dist="fixed", length=150, errors="short",
             scores="bwa", w=100, tuned=False),
        # a band wider than the 16-bit lanes take
        dict(name="wide_device", api="device", pairs=1000, dist="lognormal", length=5000, errors="ont",
             scores="ont", w=1000, tuned=False),
        # callers that may not let a library allocate
        dict(name="ont_noalloc", api="noalloc", pairs=2500, dist="lognormal", length=5000, errors="ont",
             scores="ont", w=500, tuned=False),
        # extensions with their CIGARs, long reads
        dict(name="ont_cigar", api="cigar", pairs=2000, dist="lognormal", length=5000, errors="ont",
             scores="ont", w=500, tuned=False),
        # extensions with their CIGARs, short reads
        dict(name="short_cigar", api="cigar", pairs=20000, dist="fixed", length=150, errors="short",
             scores="bwa", w=100, tuned=False),
        # the BWA-MEM variant: each extension continues a seed's score
        dict(name="short_local", api="local", pairs=100000, dist="fixed", length=150, errors="short",
             scores="bwa", w=100, tuned=False),
        # a burst of requests of 1 to 512 pairs through the server
        dict(name="ont_serve", api="serve", pairs=4096, dist="lognormal", length=5000, errors="ont",
             scores="ont", w=500, tuned=False),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the ranges the listed ones stand for."""
    while True:
        kind = rng.choice(["small", "ont", "hifi", "skewed", "short", "ont", "short"])
        if kind == "short":
            c = dict(pairs=_log(rng, 16, 200000), dist="fixed", length=rng.randint(70, 300), errors="short",
                     scores="bwa", w=rng.randint(60, 127))
            apis = ["host", "device", "cigar", "local"]
        elif kind == "small":
            c = dict(pairs=_log(rng, 16, 4096), dist="fixed", length=_log(rng, 300, 3000), errors="small",
                     scores="ont", w=rng.randint(60, 255))
            apis = ["host", "device", "cigar"]
        elif kind == "ont":
            c = dict(pairs=_log(rng, 32, 20000), dist="lognormal", length=_log(rng, 1500, 6000), errors="ont",
                     scores="ont", w=rng.choice([rng.randint(256, 511), 500, rng.randint(768, 1000)]))
            apis = ["host", "device", "cigar", "noalloc", "serve"]
        elif kind == "hifi":
            c = dict(pairs=_log(rng, 32, 5000), dist="normal", length=_log(rng, 5000, 15000), errors="hifi",
                     scores="hifi", w=rng.randint(256, 511))
            apis = ["host", "device"]
        else:
            c = dict(pairs=_log(rng, 200, 50000), dist="pareto", length=500, errors="skewed",
                     scores="ont", w=rng.randint(512, 760))
            apis = ["host", "device"]
        c["api"] = rng.choice(apis)
        c["tuned"] = False
        if c["api"] in ("cigar", "serve"):
            c["pairs"] = min(c["pairs"], 2000 if kind != "short" else 20000)
        if c["api"] == "noalloc" or c["w"] > 767:
            c["pairs"] = min(c["pairs"], 2500)
        if c["api"] == "cigar" and c["w"] > 767:
            continue
        return c


# ------------------------------------------------------------------ inputs


def _lengths(case, n, g, device):
    L, d = case["length"], case["dist"]
    if d == "fixed":
        return torch.full((n,), L, dtype=torch.int64, device=device)
    if d == "lognormal":
        x = torch.exp(torch.randn(n, generator=g, device=device, dtype=torch.float64) * 0.8 + math.log(L))
        return x.round().clamp(500, 50000).long()
    if d == "normal":
        x = torch.randn(n, generator=g, device=device, dtype=torch.float64) * (0.2 * L) + L
        return x.round().clamp(min=2000, max=3 * L).long()
    u = torch.rand(n, generator=g, device=device, dtype=torch.float64).clamp(min=1e-12)
    return (u ** (-1 / 1.5) * L).round().clamp(max=100000).long()


def _geometric(n, g, device):
    """Lengths of indels: geometric with mean 2."""
    u = torch.rand(n, generator=g, device=device, dtype=torch.float64).clamp(min=1e-12)
    return (torch.log(u) / math.log(0.5)).floor().long() + 1


def _mutate(q, q_len, errors, g):
    """Targets of concatenated queries: substitutions, insertions and
    deletions, and for a fraction of the pairs unrelated bases from a uniform
    position on."""
    sub, ins, dele, tail = errors
    dev, n, pairs = q.device, q.numel(), q_len.numel()
    pid = torch.repeat_interleave(torch.arange(pairs, device=dev), q_len)
    end = torch.cumsum(q_len, 0)
    pos = torch.arange(n, device=dev)
    u = torch.rand(n, generator=g, device=dev)
    is_sub = u < sub
    is_del = (u >= sub) & (u < sub + dele / 2)
    is_ins = (u >= sub + dele / 2) & (u < sub + dele / 2 + ins / 2)
    at = is_del.nonzero()[:, 0]
    run = torch.zeros(n, dtype=torch.int64, device=dev)
    run[at] = torch.minimum(at + _geometric(at.numel(), g, dev), end[pid[at]])
    deleted = torch.cummax(run, 0).values > pos
    at = is_ins.nonzero()[:, 0]
    extra = torch.zeros(n, dtype=torch.int64, device=dev)
    extra[at] = _geometric(at.numel(), g, dev)
    base = torch.where(is_sub, (q + torch.randint(1, 4, (n,), generator=g, device=dev, dtype=torch.uint8)) & 3, q)
    count = extra + (~deleted).long()
    src = torch.repeat_interleave(pos, count)
    out = base[src]
    within = torch.arange(src.numel(), device=dev) - (torch.cumsum(count, 0) - count)[src]
    t_pid = pid[src]
    fresh = within < extra[src]
    t_len = torch.bincount(t_pid, minlength=pairs)
    if tail > 0:
        has = torch.rand(pairs, generator=g, device=dev) < tail
        cut = (torch.rand(pairs, generator=g, device=dev, dtype=torch.float64) * t_len).floor().long()
        where = torch.arange(src.numel(), device=dev) - (torch.cumsum(t_len, 0) - t_len)[t_pid]
        fresh = fresh | (has[t_pid] & (where >= cut[t_pid]))
    rnd = torch.randint(0, 4, (out.numel(),), generator=g, device=dev, dtype=torch.uint8)
    return torch.where(fresh, rnd, out), t_len


def _pack(codes):
    """16 bases per 32-bit word, base k at bits 2k."""
    n = codes.numel()
    x = torch.zeros((n + 15) // 16 * 16 or 16, dtype=torch.int64, device=codes.device)
    x[:n] = codes
    x = (x.view(-1, 16) << (2 * torch.arange(16, device=codes.device))).sum(1)
    return torch.where(x >= 2 ** 31, x - 2 ** 32, x).to(torch.int32)


def _pairs(case, seed, device):
    """Packed streams, offsets and lengths of the case's pairs, and the seeds'
    scores of the local variant, all on `device`."""
    g = torch.Generator(device=device)
    g.manual_seed(int(seed) * 1000003 + 12345)
    n = case["pairs"]
    q_len = _lengths(case, n, g, device)
    qs, ts, tls = [], [], []
    bounds = torch.cumsum(q_len, 0).cpu()
    i = 0
    while i < n:                          # about 32 M bases at a time
        done = int(bounds[i - 1]) if i else 0
        j = max(i + 1, int(torch.searchsorted(bounds, torch.tensor(done + (1 << 25)), right=True)))
        ql = q_len[i:j]
        q = torch.randint(0, 4, (int(ql.sum()),), generator=g, device=device, dtype=torch.uint8)
        t, tl = _mutate(q, ql, ERRORS[case["errors"]], g)
        qs.append(q)
        ts.append(t)
        tls.append(tl)
        i = j
    t_len = torch.cat(tls)
    h0 = torch.randint(19, 61, (n,), generator=g, device=device, dtype=torch.int32)
    return dict(q=torch.cat(qs), t=torch.cat(ts), q_len=q_len, t_len=t_len,
                q_off=torch.cumsum(q_len, 0) - q_len, t_off=torch.cumsum(t_len, 0) - t_len, h0=h0)


def _scoring(case):
    a, b, q, e, q2, e2, z, eb = SCORES[case["scores"]]
    return Scoring(a=a, b=b, q=q, e=e, q2=q2, e2=e2, w=case["w"], zdrop=z, end_bonus=eb)


# one context for the life of the program, as a mapper keeps it: its buffers,
# captured graphs and tuned plans serve every batch
_CONTEXT = {}


def _context(tuned):
    if tuned not in _CONTEXT:
        _CONTEXT[tuned] = A.Context(0, autotune=tuned)
    return _CONTEXT[tuned]


def _host(x):
    """A numpy array in pinned memory (and the tensor that owns it)."""
    p = x.cpu().pin_memory() if DEV == "cuda" else x.cpu()
    return p.numpy()


def prepare(case, seed):
    p = _pairs(case, seed, DEV)
    s = {"api": case["api"], "scoring": _scoring(case), "n": case["pairs"]}
    arrays = dict(q_packed=_pack(p["q"]), t_packed=_pack(p["t"]), q_off=p["q_off"], t_off=p["t_off"],
                  q_len=p["q_len"].to(torch.int32), t_len=p["t_len"].to(torch.int32))
    if case["api"] in ("device", "noalloc"):
        s["args"] = arrays
        s["out"] = torch.empty(case["pairs"] * 48, dtype=torch.uint8, device=DEV)
    else:
        h = {k: _host(v) for k, v in arrays.items()}
        h["q_packed"] = h["q_packed"].view(np.uint32)
        h["t_packed"] = h["t_packed"].view(np.uint32)
        s["batch"] = A.PackedBatch(**h)
        s["h0"] = _host(p["h0"])
        s["out"] = _host(torch.zeros(case["pairs"] * 48, dtype=torch.uint8)).view(A.RESULT_DTYPE)
    if case["api"] == "serve":
        # requests of 1 to 512 pairs, together every pair of the batch
        rng = np.random.default_rng(int(seed))
        cuts, at, b = [], 0, s["batch"]
        while at < s["n"]:
            k = min(int(rng.integers(1, 513)), s["n"] - at)
            cuts.append(slice(at, at + k))
            at += k
        s["requests"] = [A.PackedBatch(b.q_packed, b.t_packed, b.q_off[c].copy(), b.t_off[c].copy(),
                                       b.q_len[c].copy(), b.t_len[c].copy()) for c in cuts]
        s["server_context"] = A.Context(0)
        s["server"] = A.Server(s["server_context"], mem_budget_bytes=2 << 30)
    elif case["api"] != "noalloc":
        if case["api"] == "cigar":
            # one buffer for the runs of every batch of this size (an indel
            # adds two runs to a pair's path)
            s["runs"] = np.zeros(int(case["pairs"] * (16 + 0.25 * np.mean(_mean_lengths(case)))) + 20000, np.uint32)
        s["ctx"] = _context(bool(case["tuned"]))
        if case["tuned"]:
            # the first host batch of a scoring lets the context choose its plan
            if s["ctx"].tune_variants(s["scoring"]) is None:
                s["ctx"].align_host(s["batch"], s["scoring"])
    if DEV == "cuda":
        torch.cuda.synchronize()
    return s


def _host_records(r):
    v = r.view(np.int32).reshape(-1, 12)
    u = r.view(np.uint8).reshape(-1, 48)
    return {"scores": v[:, :8], "cells": r["cells"], "stops": u[:, 40:42], "lane16": u[:, 42]}


def _device_records(out):
    u = out.view(-1, 48)
    return {"scores": u[:, :32].view(torch.int32), "cells": u[:, 32:40].view(torch.int64)[:, 0],
            "stops": u[:, 40:42], "lane16": u[:, 42]}


def run(state):
    s, api = state, state["api"]
    if api == "device":
        s["ctx"].align_device(out=s["out"], scoring=s["scoring"], **s["args"])
        return _device_records(s["out"])
    if api == "noalloc":
        A.agatha_align_batch_noalloc(out=s["out"], scoring=s["scoring"], **s["args"])
        return _device_records(s["out"])
    if api == "host":
        return _host_records(s["ctx"].align_host(s["batch"], s["scoring"], out=s["out"]))
    if api == "local":
        return _host_records(s["ctx"].align_local(s["batch"], s["scoring"], s["h0"], out=s["out"]))
    if api == "cigar":
        res, off, cigar = s["ctx"].align_cigar(s["batch"], s["scoring"])
        s["runs"][:cigar.shape[0]] = cigar
        return {**_host_records(res), "offsets": off, "cigar": s["runs"]}
    srv = s["server"]
    tickets = [srv.submit(r, s["scoring"]) for r in s["requests"]]
    return _host_records(np.concatenate([srv.wait(t) for t in tickets]))


# ------------------------------------------------------------------- work


def _mean_lengths(case):
    """Read lengths of the case's distribution, evenly over its quantiles."""
    u = (np.arange(512) + 0.5) / 512
    L, d = case["length"], case["dist"]
    if d == "fixed":
        return np.full(1, float(L))
    if d == "pareto":
        return np.minimum(L * (1 - u) ** (-1 / 1.5), 100000)
    z = math.sqrt(2) * torch.erfinv(torch.from_numpy(2 * u - 1)).numpy()
    if d == "lognormal":
        return np.clip(L * np.exp(0.8 * z), 500, 50000)
    return np.clip(L + 0.2 * L * z, 2000, 3 * L)


def work(case):
    """Packed bases and lengths read once, records (and runs) written once; 13
    integer operations for each band cell of a two-piece extension (7 with one
    piece), and 9 more where the path is wanted."""
    L = _mean_lengths(case)
    n, w = case["pairs"], case["w"]
    tail = ERRORS[case["errors"]][3]
    # a divergent tail stops the extension about halfway on average
    reach = L * (1 - tail / 2)
    band = np.where(L > w, (2 * w + 1.0) * reach - w * (w + 1.0), reach * reach)
    cells = float(np.mean(band)) * n
    ops = 13 if SCORES[case["scores"]][4] > SCORES[case["scores"]][2] else 7
    if case["api"] == "cigar":
        ops += 9
    moved = n * (2 * float(np.mean(L)) / 4 + 24 + 48)
    if case["api"] == "cigar":
        errors = sum(ERRORS[case["errors"]][:3])
        moved += 4 * n * (1 + errors * float(np.mean(L)))
    return {"bytes": moved, "flops": ops * cells}


# ------------------------------------------------------------------ exact


def exact(case, seed):
    """The extension's definition on all pairs at once, anti-diagonal by
    anti-diagonal, in 64-bit integers (fixed-length batches of moderate size;
    not the local variant, and no paths)."""
    if case["api"] not in ("host", "device") or case["dist"] != "fixed":
        return None
    if case["pairs"] * (2 * case["w"] + 3) > 1 << 26 or case["length"] > 3000:
        return None
    p = _pairs(case, seed, DEV)
    a, b, q, e, q2, e2, zdrop, bonus = SCORES[case["scores"]]
    w, n, dev = case["w"], case["pairs"], p["q"].device
    NEG = -(1 << 40)
    i64 = dict(dtype=torch.int64, device=dev)
    ql, tl = p["q_len"][:, None], p["t_len"][:, None]
    w = min(w, int(torch.maximum(p["q_len"], p["t_len"]).max()))
    d = torch.arange(-w - 1, w + 2, device=dev)[None, :]          # t - q
    width = d.shape[1]

    def gap(x):
        return torch.minimum(q + x * e, q2 + x * e2)

    def virtual(r):
        """Virtual row and column cells of anti-diagonal r, NEG elsewhere."""
        H = torch.full((n, width), NEG, **i64)
        if r >= -2:
            t, s = (r + d) // 2, (r - d) // 2
            on = ((r + d) % 2 == 0) & (((t == -1) & (s >= -1)) | ((s == -1) & (t >= -1)))
            on = on & (t < tl) & (s < ql)
            cost = torch.where((t == -1) & (s == -1), torch.zeros_like(t), -gap(torch.maximum(t, s) + 1))
            H = torch.where(on, cost.expand(n, width), H)
        return H

    def left(x):                                                   # value at d - 1
        return torch.nn.functional.pad(x[:, :-1], (1, 0), value=NEG)

    def right(x):                                                  # value at d + 1
        return torch.nn.functional.pad(x[:, 1:], (0, 1), value=NEG)

    H2, H1 = virtual(-2), virtual(-1)
    none = torch.full((n, width), NEG, **i64)
    E, F, G, K = (torch.maximum(none, H1 - c) for c in (q + e, q + e, q2 + e2, q2 + e2))
    best = torch.zeros(n, **i64)
    bt, bq = torch.full((n,), -1, **i64), torch.full((n,), -1, **i64)
    lowest = int(A.NEG_INF)
    mqe, mte, gs = (torch.full((n,), lowest, **i64) for _ in range(3))
    mqe_t, mte_q = torch.full((n,), -1, **i64), torch.full((n,), -1, **i64)
    cells, drop = torch.zeros(n, **i64), torch.zeros(n, dtype=torch.bool, device=dev)
    alive = torch.ones(n, dtype=torch.bool, device=dev)
    last = (ql + tl - 2)[:, 0]
    limit = p["t"].numel() - 1
    qlimit = p["q"].numel() - 1
    for r in range(int(last.max()) + 1):
        alive = alive & (last >= r)
        t, s = (r + d) // 2, (r - d) // 2
        real = ((r + d) % 2 == 0) & (d.abs() <= w) & (t >= 0) & (s >= 0) & (t < tl) & (s < ql)
        tb = p["t"][(p["t_off"][:, None] + t).clamp(0, limit)]
        qb = p["q"][(p["q_off"][:, None] + s).clamp(0, qlimit)]
        S = torch.where(tb == qb, a, -b)
        Ei, Fi, Gi, Ki = left(E), right(F), left(G), right(K)
        H = torch.maximum(torch.maximum(torch.maximum(H2 + S, Ei), torch.maximum(Fi, Gi)), Ki)
        H = torch.where(real, H, NEG)
        count = real.sum(1)
        gone = alive & (count == 0)
        drop = drop | gone
        alive = alive & ~gone
        cells = cells + torch.where(alive, count, 0)
        # the last query column and target row
        for at, value, place, other in ((s == ql - 1, "mqe", "mqe_t", t), (t == tl - 1, "mte", "mte_q", s)):
            v = torch.where(real & at, H, lowest).max(1).values
            where = torch.where(real & at, other, -1).max(1).values
            if value == "mqe":
                better = alive & (v > mqe)
                mqe, mqe_t = torch.where(better, v, mqe), torch.where(better, where, mqe_t)
            else:
                better = alive & (v > mte)
                mte, mte_q = torch.where(better, v, mte), torch.where(better, where, mte_q)
        m = H.max(1).values
        first = torch.where(H == m[:, None], d.expand(n, width), 1 << 30).min(1).values
        mt, mq = (r + first) // 2, (r - first) // 2
        up = alive & (m > best)
        stop = torch.zeros_like(alive)
        if zdrop >= 0:
            stop = alive & ~up & (mt >= bt) & (mq >= bq) & (best - m > zdrop + ((mt - bt) - (mq - bq)).abs() * e2)
        best, bt, bq = torch.where(up, m, best), torch.where(up, mt, bt), torch.where(up, mq, bq)
        drop = drop | stop
        alive = alive & ~stop
        corner = torch.where(real & (t == tl - 1) & (s == ql - 1), H, lowest).max(1).values
        gs = torch.where(alive & (last == r), corner, gs)
        if not bool(alive.any()):
            break
        H = torch.maximum(H, virtual(r)) if r <= w else H
        E, F = torch.maximum(Ei - e, H - q - e), torch.maximum(Fi - e, H - q - e)
        G, K = torch.maximum(Gi - e2, H - q2 - e2), torch.maximum(Ki - e2, H - q2 - e2)
        floor = NEG // 2
        E, F, G, K = (torch.where(x < floor, NEG, x) for x in (E, F, G, K))
        # a state leaves real and virtual cells only
        keep = H > floor
        E, F, G, K = (torch.where(keep, x, NEG) for x in (E, F, G, K))
        H2, H1 = H1, H
    reach = ~drop & (mqe != lowest) & (mqe + bonus > best)
    scores = torch.stack([best, bq, bt, gs, mqe, mqe_t, mte, mte_q], 1).to(torch.int32)
    out = {"scores": scores, "cells": cells, "stops": torch.stack([drop, reach], 1).to(torch.uint8),
           "lane16": None}
    if case["api"] == "host":
        out = {k: None if v is None else v.cpu().numpy() for k, v in out.items()}
    return out
