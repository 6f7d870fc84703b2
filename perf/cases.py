"""The work that a user of the aligner has it do, case by case, through its public entry points.

A case is a dict of plain values: the entry point (`entry`), the algorithm, the number of pairs and the shape of
their sequences (lengths log-uniform in len_lo .. len_hi, edit rates uniform in rate_lo .. rate_hi, a share of
unrelated pairs), the costs, the threshold (max_edits, or ceil(frac * read length) per pair when frac > 0) and the
options.  Reads are uniform random DNA; a target is its read with substitutions, insertions and deletions in equal
parts at random positions, or, for an unrelated pair, independent DNA of the read's length.
"""
import math

import numpy as np
import torch

import paper_2208_01243_gb300 as aim

BASE = {"entry": "plain", "algo": "wfa", "pairs": 0, "len_lo": 150, "len_hi": 150, "rate_lo": 0.04, "rate_hi": 0.04,
        "unrelated": 0.0, "mismatch": 4, "gap_open": 6, "gap_extend": 2, "max_edits": 6, "frac": 0.0, "band": -1,
        "cigars": True, "packed": False, "requests": 0, "workspace_gib": 4.0}


def _case(**kw):
    c = dict(BASE)
    c.update(kw)
    return c


def listed():
    return [
        # one small batch of short reads as an interactive caller sends it: launches and latency
        _case(name="wfa_150bp_61", pairs=61, unrelated=0.10, workspace_gib=0.25),
        # the smallest throughput shape: edit distance of 100 bp reads, at most 10 edits
        _case(name="edit_100bp_10k", algo="edit", pairs=10_000, len_lo=100, len_hi=100, rate_lo=0.02, rate_hi=0.02,
              mismatch=1, gap_open=0, gap_extend=1, max_edits=10, workspace_gib=1.0),
        # read mapping's verification step: 150 bp reads against candidates, a tenth of them unrelated and rejected
        _case(name="wfa_150bp_1M", pairs=1_000_003, unrelated=0.10),
        # banded gap-affine DP over 250 bp reads with 10 % errors
        _case(name="gotoh_250bp_1M", algo="gotoh", pairs=1_000_000, len_lo=250, len_hi=250, rate_lo=0.10, rate_hi=0.10,
              max_edits=25, band=25),
        # reads of uneven length and quality, planned once and replayed
        _case(name="wfa_uneven_1M", entry="batch", pairs=1_000_000, len_lo=100, len_hi=1000, rate_lo=0.01,
              rate_hi=0.10, frac=0.10, workspace_gib=16.0),
        # long reads, planned once and replayed
        _case(name="wfa_long_4k", entry="batch", pairs=4_000, len_lo=2000, len_hi=10_000, rate_lo=0.01, rate_hi=0.10,
              frac=0.10, workspace_gib=16.0),
        # the heuristic wavefront on 1,000 bp reads with 5 % errors
        _case(name="adaptive_1000bp_200k", algo="wfa_adaptive", pairs=200_000, len_lo=1000, len_hi=1000, rate_lo=0.05,
              rate_hi=0.05, mismatch=3, gap_open=4, gap_extend=1, max_edits=50),
        # windowed bitap on short reads ...
        _case(name="genasm_150bp_1M", algo="genasm", pairs=1_000_000, rate_lo=0.05, rate_hi=0.05, mismatch=1,
              gap_open=0, gap_extend=1, max_edits=8),
        # ... and over many windows of longer ones
        _case(name="genasm_1000bp_200k", algo="genasm", pairs=200_000, len_lo=1000, len_hi=1000, rate_lo=0.05,
              rate_hi=0.05, mismatch=1, gap_open=0, gap_extend=1, max_edits=50),
        # a program that holds its reads in host memory: the transfers are part of the call
        _case(name="host_150bp_500k", entry="host", pairs=500_009, unrelated=0.10),
        # packing a read set of uneven lengths back to back, before it is aligned many times
        _case(name="pack_uneven_1M", entry="pack", pairs=1_000_000, len_lo=100, len_hi=1000),
        # a server's burst: requests of 1 to 4,096 pairs of 100 to 10,000 bp, all submitted, then awaited
        _case(name="serve_24", entry="serve", pairs=0, requests=24, len_lo=100, len_hi=10_000, rate_lo=0.01,
              rate_hi=0.10, frac=0.10, workspace_gib=16.0),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(math.exp(rng.uniform(math.log(lo), math.log(hi + 1))))))


def draw(rng):
    """One more case: any entry point and algorithm, sizes spread over their logarithms, odd ones among them."""
    kind = rng.choice(["wfa", "wfa", "wfa_band", "edit", "gotoh", "adaptive", "genasm", "genasm", "batch", "batch",
                       "long", "host", "pack", "serve", "static"])
    if kind in ("wfa", "wfa_band", "host", "static"):
        n = _log_int(rng, 80, 320)
        edits = _log_int(rng, 2, max(3, n // 12))
        kw = dict(pairs=_log_int(rng, 16, 150_000_000 // n // max(1, edits // 8)), len_lo=n, len_hi=n,
                  max_edits=edits, rate_lo=0.7 * edits / n, rate_hi=0.7 * edits / n,
                  unrelated=rng.choice([0.0, 0.1]), cigars=rng.random() < 0.8)
        if kind == "wfa_band":
            kw["band"] = rng.randint(5, 30)
        if kind == "wfa":
            kw["packed"] = rng.random() < 0.5
            kw["mismatch"], kw["gap_open"], kw["gap_extend"] = rng.choice([(4, 6, 2), (4, 6, 2), (3, 4, 1)])
        if kind == "static":
            kw.update(entry="static", packed=True, pairs=min(kw["pairs"], 300_000), workspace_gib=0.0)
        if kind == "host":
            kw.update(entry="host", pairs=max(1000, kw["pairs"] // 2))
        return _case(**kw)
    if kind in ("edit", "gotoh"):
        n = _log_int(rng, 60, 260)
        edits = rng.randint(3, max(4, n // 10))
        kw = dict(algo=kind, len_lo=n, len_hi=n, max_edits=edits, rate_lo=0.7 * edits / n, rate_hi=0.7 * edits / n,
                  packed=rng.random() < 0.3)
        if kind == "edit":
            kw.update(mismatch=1, gap_open=0, gap_extend=1, pairs=_log_int(rng, 100, 100_000_000 // n))
        else:
            kw.update(band=min(31, edits), pairs=_log_int(rng, 100, 100_000_000 // n))
        return _case(**kw)
    if kind == "adaptive":
        n = _log_int(rng, 120, 5000)
        pct = rng.choice([0.02, 0.05])
        return _case(algo="wfa_adaptive", pairs=_log_int(rng, 50, 100_000_000 // n), len_lo=n, len_hi=n, rate_lo=pct,
                     rate_hi=pct, mismatch=3, gap_open=4, gap_extend=1, max_edits=math.ceil(pct * n))
    if kind == "genasm":
        n = _log_int(rng, 80, 1500)
        pct = rng.choice([0.01, 0.05])
        return _case(algo="genasm", pairs=_log_int(rng, 100, 150_000_000 // n), len_lo=n, len_hi=n, rate_lo=pct,
                     rate_hi=pct, mismatch=1, gap_open=0, gap_extend=1, max_edits=math.ceil(pct * n))
    if kind == "batch":
        lo = _log_int(rng, 80, 300)
        hi = _log_int(rng, 2 * lo, 1000)
        return _case(entry="batch", pairs=_log_int(rng, 2000, 250_000_000 // hi), len_lo=lo, len_hi=hi, rate_lo=0.01,
                     rate_hi=0.10, frac=0.10, workspace_gib=8.0)
    if kind == "long":
        lo = _log_int(rng, 1500, 4000)
        return _case(entry="batch", pairs=_log_int(rng, 64, 3000), len_lo=lo, len_hi=_log_int(rng, lo, 10_000),
                     rate_lo=0.01, rate_hi=0.10, frac=0.10, workspace_gib=16.0)
    if kind == "pack":
        lo = _log_int(rng, 30, 2000)
        hi = _log_int(rng, lo, 10_000)
        return _case(entry="pack", pairs=_log_int(rng, 100, 350_000_000 // hi), len_lo=lo, len_hi=hi)
    return _case(entry="serve", requests=rng.randint(3, 20), len_lo=100, len_hi=_log_int(rng, 300, 8000),
                 rate_lo=0.01, rate_hi=0.10, frac=0.10, workspace_gib=16.0)


# ---------------------------------------------------------------- inputs

def _log_uniform(g, n, lo, hi):
    """n whole numbers log-uniform in lo .. hi: the distribution's n quantiles in an order of the seed's own, so that
    their sum, and with it the size of every array laid out from them, is the same for every seed."""
    u = (torch.randperm(n, generator=g, device="cuda").double() + 0.5) / n
    return torch.exp(math.log(lo) + u * math.log((hi + 1) / lo)).floor().long().clamp_(lo, hi)


def _lengths(c, g, n):
    return _log_uniform(g, n, c["len_lo"], c["len_hi"])


def _starts(lens):
    off = torch.zeros(lens.numel() + 1, dtype=torch.int64, device=lens.device)
    off[1:] = torch.cumsum(lens, 0)
    return off


def _pairs(c, g, n):
    """n read/target pairs as ASCII laid out back to back on the device, with offsets and lengths."""
    dev = "cuda"
    rl = _lengths(c, g, n)
    roff = _starts(rl)
    total = int(roff[-1])
    read = torch.randint(0, 4, (total,), generator=g, device=dev, dtype=torch.uint8)
    unrelated = torch.rand(n, generator=g, device=dev) < c["unrelated"]
    rate = c["rate_lo"] + (c["rate_hi"] - c["rate_lo"]) * torch.rand(n, generator=g, device=dev)
    edits = (rate * rl + 0.5).floor().long().masked_fill_(unrelated, 0)
    # one code per read base: 0 kept, 1 deleted, 2..4 substituted, 5..8 a base inserted before it; of several edits
    # on one base the largest code stays
    who = torch.repeat_interleave(torch.arange(n, device=dev), edits)
    k = who.numel()
    at = roff[:-1][who] + (torch.rand(k, generator=g, device=dev, dtype=torch.float64) * rl[who]).long()
    what = torch.randint(0, 3, (k,), generator=g, device=dev)
    code = torch.where(what == 0, 1, torch.where(what == 1, 2 + torch.randint(0, 3, (k,), generator=g, device=dev),
                                                 5 + torch.randint(0, 4, (k,), generator=g, device=dev)))
    op = torch.zeros(total, dtype=torch.int32, device=dev)
    op.scatter_reduce_(0, at, code.int(), "amax")
    op = op.to(torch.uint8)
    del who, at, what, code
    count = torch.ones(total, dtype=torch.uint8, device=dev)
    count[op == 1] = 0
    count[op >= 5] = 2
    end = torch.cumsum(count, 0, dtype=torch.int64)
    tend = torch.zeros(n + 1, dtype=torch.int64, device=dev)
    tend[1:] = end[roff[1:] - 1]
    base = torch.where((op >= 2) & (op <= 4), (read + op - 1) & 3, read)
    if c["unrelated"] > 0:
        fresh = torch.randint(0, 4, (total,), generator=g, device=dev, dtype=torch.uint8)
        base = torch.where(torch.repeat_interleave(unrelated, rl), fresh, base)
    target = torch.empty(int(tend[-1]), dtype=torch.uint8, device=dev)
    kept = count > 0
    target[end[kept] - 1] = base[kept]
    put = op >= 5
    target[end[put] - 2] = op[put] - 5
    letters = torch.tensor(list(b"ACGT"), dtype=torch.uint8, device=dev)

    def ascii_of(x):
        y = torch.empty_like(x)
        for b in range(4):
            y[x == b] = letters[b]
        return y
    tl = tend[1:] - tend[:-1]
    return {"reads": ascii_of(read), "targets": ascii_of(target), "ro": roff[:-1].contiguous(),
            "to": tend[:-1].contiguous(), "rl": rl.int(), "tl": tl.int()}


def _thresholds(c, p):
    """(largest threshold, thresholds per pair or None)."""
    if c["frac"] > 0:
        me = torch.ceil(c["frac"] * p["rl"].double() - 1e-9).int()
        return int(me.max()), me
    return c["max_edits"], None


def _unit(c):
    return c["algo"] in ("edit", "genasm")


def _cigar_offsets(c, p, me):
    """Room for every CIGAR that the threshold admits: an edit run costs at least the cheapest edit, runs alternate."""
    lim = (me.long() if me is not None else torch.full_like(p["rl"], c["max_edits"]).long())
    if not _unit(c):
        first = c["gap_open"] + c["gap_extend"]
        lim = lim * max(c["mismatch"], first) // min(c["mismatch"], first)
    return _starts(torch.minimum(2 * lim + 1, p["rl"].long() + p["tl"].long() + 1))


def _costs(c):
    return aim.penalties(c["mismatch"], c["gap_open"], c["gap_extend"], band=c["band"])


class _Plan:
    """A batch plan and its aligner, given back together."""

    def __init__(self, al, plan):
        self.al, self.plan = al, plan

    def __del__(self):
        aim.aim_batch_destroy(self.plan)
        self.al.close()


class _Server:
    def __init__(self, al, server):
        self.al, self.server = al, server

    def __del__(self):
        aim.aim_server_destroy(self.server)
        self.al.close()


def _pinned(t):
    h = torch.empty(t.shape, dtype=t.dtype, pin_memory=True)
    h.copy_(t)
    return h.numpy()


def _outputs(n, runs, dev="cuda"):
    pin = dev == "cpu"
    z = lambda k, dt: torch.zeros(max(k, 1), dtype=dt, device=dev, pin_memory=pin)  # noqa: E731
    return {"scores": z(n, torch.int32), "flags": z(n, torch.uint8), "lens": z(n, torch.int32),
            "cigars": z(runs, torch.int32) if runs else None}


def _pack_offsets(lens):
    return _starts((lens.long() + 31) // 32)


def prepare(case, seed):
    c = dict(BASE, **case)
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    s = {"c": c, "pen": _costs(c)}
    if c["entry"] == "pack":
        rl = _lengths(c, g, c["pairs"])
        off, woff = _starts(rl), _pack_offsets(rl)
        letters = torch.tensor(list(b"ACGT"), dtype=torch.uint8, device="cuda")
        s["ascii"] = letters[torch.randint(0, 4, (int(off[-1]),), generator=g, device="cuda", dtype=torch.int32)]
        s.update(al=aim.Aligner(0, 1 << 20), off=off[:-1].contiguous(), lens=rl.int(), woff=woff[:-1].contiguous(),
                 words=torch.zeros(int(woff[-1]), dtype=torch.int64, device="cuda"),
                 bad=torch.zeros(c["pairs"], dtype=torch.uint8, device="cuda"))
        return s
    if c["entry"] == "serve":
        sizes = _log_uniform(g, c["requests"], 1, 4096).tolist()
        n = sum(sizes)
        p = _pairs(c, g, n)
        _, me = _thresholds(c, p)
        coff = _cigar_offsets(c, p, me)
        h = {k: v.cpu().numpy() for k, v in p.items()}
        me, coff = me.cpu().numpy(), coff.cpu().numpy()
        out = {"scores": np.zeros(n, np.int32), "flags": np.zeros(n, np.uint8), "lens": np.zeros(n, np.int32),
               "cigars": np.zeros(int(coff[-1]), np.int32)}
        s["out"], s["requests"], at = out, [], 0
        for k in sizes:
            b = at + k
            r0, r1 = int(h["ro"][at]), int(h["ro"][b - 1] + h["rl"][b - 1])
            t0, t1 = int(h["to"][at]), int(h["to"][b - 1] + h["tl"][b - 1])
            c0, c1 = int(coff[at]), int(coff[b])
            s["requests"].append((h["reads"][r0:r1], h["targets"][t0:t1], (h["ro"][at:b] - r0).astype(np.uint64),
                                  (h["to"][at:b] - t0).astype(np.uint64), h["rl"][at:b].view(np.uint32),
                                  h["tl"][at:b].view(np.uint32), me[at:b], out["scores"][at:b], out["flags"][at:b],
                                  out["lens"][at:b], out["cigars"][c0:c1], (coff[at:b + 1] - c0).astype(np.uint64)))
            at = b
        al = aim.Aligner(0, 1 << 20)
        s["server"] = _Server(al, aim.aim_server_create(al.ctx, s["pen"], int(c["workspace_gib"] * 2**30), 512 << 20))
        return s
    p = _pairs(c, g, c["pairs"])
    s["max_edits"], me = _thresholds(c, p)
    s["max_length"] = int(torch.maximum(p["rl"].max(), p["tl"].max()))
    coff = _cigar_offsets(c, p, me) if c["cigars"] else None
    runs = int(coff[-1]) if coff is not None else 0
    if c["entry"] == "host":
        s["al"] = aim.Aligner(0, int(c["workspace_gib"] * 2**30))
        s["in"] = {k: _pinned(v) for k, v in p.items()}
        s["me"] = _pinned(me) if me is not None else None
        s["coff"] = _pinned(coff).view(np.uint64) if coff is not None else None
        s["out"] = {k: v.numpy() if v is not None else None for k, v in _outputs(c["pairs"], runs, "cpu").items()}
        return s
    s.update(p=p, me=me, coff=coff, out=_outputs(c["pairs"], runs))
    o = s["out"]
    if c["entry"] == "batch":
        al = aim.Aligner(0, 64 << 20)
        plan = aim.aim_batch_plan(al.ctx, p["reads"], p["targets"], p["ro"], p["to"], p["rl"], p["tl"],
                                  s["max_length"], s["pen"], s["max_edits"], me, o["scores"], o["cigars"], coff,
                                  o["lens"], o["flags"], scratch_bytes=int(c["workspace_gib"] * 2**30), autotune=True)
        s["plan"] = _Plan(al, plan)
        return s
    s["al"] = aim.Aligner(0, int(c["workspace_gib"] * 2**30) or 1 << 20)
    if c["packed"]:
        for q, off in (("reads", "ro"), ("targets", "to")):
            lens = p["rl" if q == "reads" else "tl"]
            woff = _pack_offsets(lens)
            words = torch.zeros(int(woff[-1]), dtype=torch.int64, device="cuda")
            aim.aim_pack_2bit(s["al"].ctx, p[q], p[off], lens, words, woff[:-1].contiguous())
            torch.cuda.synchronize()
            p[q], p[off] = words, woff[:-1].contiguous()
    return s


def run(s):
    c = s["c"]
    if c["entry"] == "pack":
        aim.aim_pack_2bit(s["al"].ctx, s["ascii"], s["off"], s["lens"], s["words"], s["woff"], s["bad"])
        return {"words": s["words"], "bad": s["bad"]}
    o = s["out"]
    if c["entry"] == "serve":
        server = s["server"].server
        tickets = [aim.aim_server_submit(server, r, t, ro, to, rl, tl, me, sc, fl, le, ci, co)
                   for r, t, ro, to, rl, tl, me, sc, fl, le, ci, co in s["requests"]]
        for ticket, _ in tickets:
            aim.aim_server_wait(server, ticket)
    elif c["entry"] == "host":
        h = s["in"]
        aim.aim_align_batch_host(s["al"].ctx, h["reads"], h["targets"], h["ro"], h["to"], h["rl"], h["tl"],
                                 s["max_length"], c["algo"], s["pen"], s["max_edits"], s["me"], o["scores"],
                                 o["cigars"], s["coff"], o["lens"], o["flags"])
    elif c["entry"] == "batch":
        aim.aim_batch_run(s["plan"].plan)
    else:
        p = s["p"]
        seqs = (p["reads"], p["targets"], p["ro"], p["to"], p["rl"], p["tl"], s["max_length"])
        rest = (s["pen"], s["max_edits"], s["me"], o["scores"], o["cigars"], s["coff"], o["lens"], o["flags"])
        if c["entry"] == "static":
            aim.aim_wfa_align_static(*seqs, *rest)
        else:
            f = aim.aim_align_batch if c["packed"] else aim.aim_align_batch_ascii
            f(s["al"].ctx, *seqs, c["algo"], *rest)
    return {"scores": o["scores"], "flags": o["flags"], "lens": o["lens"], "cigars": o["cigars"]}


def _mean_length(c):
    lo, hi = c["len_lo"], c["len_hi"]
    return float(lo) if lo == hi else (hi - lo) / math.log(hi / lo)


def work(case):
    """Bytes: the sequences, offsets, lengths and thresholds once, the scores, flags, run counts and a run or two
    per edit once.  Operations: integer operations of the cells or wavefront entries that the algorithm computes
    for the pairs' own edits (a wavefront of score s and cost step e holds about s / e diagonals; a banded DP its
    band; bitap one 64-bit word per target base and edit of a window)."""
    c = dict(BASE, **case)
    n = c["pairs"] if c["entry"] != "serve" else c["requests"] * 4095 / math.log(4096)
    length = _mean_length(c)
    rate = (c["rate_lo"] + c["rate_hi"]) / 2
    if c["entry"] == "pack":
        return {"bytes": n * (length + 8 * (length + 31) / 32 + 21), "flops": 0.0}
    edits = rate * length
    seq = 2 * length / (4 if c["packed"] else 1)
    data = n * (seq + 24 + (4 if c["frac"] > 0 else 0) + 9 + (8 + 4 * (2 * edits + 1) if c["cigars"] else 0))
    if c["algo"] in ("edit", "gotoh"):
        band = c["max_edits"] if c["band"] < 0 else min(c["band"], c["max_edits"] * 4)
        ops = length * (2 * band + 1) * (5 if c["algo"] == "edit" else 14)
    elif c["algo"] == "genasm":
        ops = length * 64 / 40 * (1 + rate * 64) * 16
    else:
        unit = math.gcd(math.gcd(c["mismatch"], c["gap_open"]), c["gap_extend"])
        per_edit = (c["mismatch"] + 2 * (c["gap_open"] + c["gap_extend"])) / 3 / unit
        # the mean of (edits)^2 over the drawn lengths and rates, not the square of the mean
        lo, hi = c["len_lo"], c["len_hi"]
        len2 = length * length if lo == hi else (hi * hi - lo * lo) / 2 / math.log(hi / lo)
        a, b = c["rate_lo"], c["rate_hi"]
        edits2 = len2 * (a * a + a * b + b * b) / 3
        entries = edits2 * per_edit * per_edit / 2 / (c["gap_extend"] / unit)
        ops = entries * (6 + 12) + length / 32 * 12
    return {"bytes": data, "flops": n * ops}


# ---------------------------------------------------------------- what the scores are, by plain dynamic programming

def _dp_scores(p, c, limit, band):
    """Optimal gap-affine costs, row by row over all pairs of one batch, in 64 bits (cost above limit: -1)."""
    x, o, e = c["mismatch"], c["gap_open"], c["gap_extend"]
    n, m = p["rl"].long(), p["tl"].long()
    rows, cols, k = int(n.max()), int(m.max()), n.numel()
    inf = 1 << 40
    h = torch.arange(cols + 1, device="cuda")
    tidx = (p["to"][:, None] + h[None, :-1]).clamp_(max=p["targets"].numel() - 1)
    t = p["targets"][tidx]
    best = torch.where(h == 0, 0, o + e * h)[None, :].repeat(k, 1)
    if band >= 0:
        best[:, h > band] = inf
    ins = torch.full((k, cols + 1), inf, device="cuda", dtype=torch.int64)
    end = torch.where(n == 0, best.gather(1, m[:, None])[:, 0], inf)
    for v in range(1, rows + 1):
        base = p["reads"][(p["ro"] + v - 1).clamp(max=p["reads"].numel() - 1)]
        ins = torch.minimum(ins + e, best + o + e)
        now = ins.clone()
        now[:, 1:] = torch.minimum(now[:, 1:], best[:, :-1] + x * (t != base[:, None]))
        if band >= 0:
            out = (h - v).abs() > band
            now[:, out] = inf
            ins[:, out] = inf
        gap = torch.cummin(now + o - e * h, 1).values + e * h
        gap = torch.nn.functional.pad(gap[:, :-1] + e, (1, 0), value=inf)
        if band >= 0:
            gap[:, out] = inf
        best = torch.minimum(now, gap)
        end = torch.where(n == v, best.gather(1, m[:, None])[:, 0], end)
    return torch.where(end > limit, -1, end)


def exact(case, seed):
    c = dict(BASE, **case)
    if c["algo"] not in ("edit", "gotoh", "wfa") or c["entry"] == "pack" or c["frac"] > 0 or \
            c["pairs"] * _mean_length(c) ** 2 > 3e10:
        return None   # the heuristics have no closed value; the large uneven batches would take minutes
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    p = _pairs(c, g, c["pairs"])
    limit = c["max_edits"] * (1 if _unit(c) else max(c["mismatch"], c["gap_open"] + c["gap_extend"]))
    scores = []
    for a in range(0, c["pairs"], 50_000):
        part = {k: v if k in ("reads", "targets") else v[a:a + 50_000] for k, v in p.items()}
        scores.append(_dp_scores(part, c, limit, c["band"]))
    scores = torch.cat(scores)
    cut = (p["tl"].long() - p["rl"].long()).abs() > c["band"] if c["band"] >= 0 else torch.zeros_like(scores).bool()
    scores = torch.where(cut, -1, scores).int()
    return {"scores": scores, "flags": (scores < 0).to(torch.uint8), "lens": None, "cigars": None}
