"""Performance cases of the framework: what a read mapper has it do, through its public entry points.

A mapper loads its reference indexes once, then sends it batches of reads: SMEM search finds exact matches, suffix
array lookup turns their intervals into positions, seed extension aligns the rest of each read around them.  The cases
are those calls, from a handful of pairs to the largest batch the framework is benchmarked on, with short and long
reads, device and host inputs, reads with N bases, scorings that need 8-bit and 16-bit scores, and the serving loop.

Every output is a whole number and has to be the same bit for bit.
"""
import functools
import math

import numpy as np
import torch

from paper_1907_12931_gb300 import bsw
from paper_1907_12931_gb300 import workload

BUDGET = 16 << 30
REF_BASES = 1 << 24           # reference the extension pairs are drawn from
FM_BASES = 16_000_000         # reference prefix indexed for the SMEM search (a 32 Mbp text)
SA_ENTRIES = 64_000_001       # suffix array of a 64 Mbp reference prefix

# kind -> what the numbers of a case mean:
#   reads   pairs of queries left and right of a random seed in read_len-base reads (0.1% SNPs and 1% errors at 151
#           bases, else 2% divergence, a tenth of it indels); target = query + w; h0 = the seed's score
#   plain   queries of 1-130 bases, 1% substitutions, a few short indels; h0 19-60
#   long    queries log-uniform 1..read_len bases with 12% error, half of it indels; w 500
#   seeds   bsw_extend_seeds: n reads of read_len bases, two seeds each, both sides extended, results filtered
#   smem    bsw_smem: n reads, every other one from the reverse strand
#   sal     bsw_sal_lookup: n intervals of geometric length
#   serve   n pairs in requests of mixed sizes, submitted together and collected
# host: inputs and results in host memory.  n_rate: share of query bases that are N.  match: match score; the other
# costs are scaled with it, as BWA-MEM's -A option does.


def _case(kind, n, read_len, host=False, n_rate=0.0, match=1, name=None):
    c = {"kind": kind, "n": int(n), "read_len": int(read_len), "host": bool(host), "n_rate": float(n_rate),
         "match": int(match)}
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # one read's worth of candidate seeds extended on their own: latency, launches
        _case("reads", 97, 151, name="reads151_97"),
        # the repository's parity configuration: a small batch of short queries
        _case("plain", 10_000, 130, name="plain_10k"),
        # a whole batch of 151 bp reads, resident on the device
        _case("reads", 2_000_000, 151, name="reads151_2m"),
        # 250 bp reads: the benchmark's headline batch, the largest
        _case("reads", 4_000_000, 250, name="reads250_4m"),
        # reads with no-calls, reference with N runs
        _case("reads", 1_000_000, 250, n_rate=0.001, name="reads250_n_1m"),
        # match 2 (mapper option -A 2): most scores pass 255
        _case("reads", 1_000_000, 250, match=2, name="reads250_match2_1m"),
        # long noisy queries, plan as the autotuner picks it for them
        _case("long", 20_000, 10_000, name="long10k_20k"),
        # the same extension as one call on host buffers: check, copies, kernels, results back
        _case("reads", 500_001, 250, host=True, name="reads250_host_500k"),
        # the seed-extension driver, reads and seeds from the host
        _case("seeds", 100_000, 151, host=True, name="seeds151_100k"),
        # seeding: SMEMs of a read batch
        _case("smem", 200_000, 151, host=True, name="smem151_200k"),
        # positions of the SMEMs' intervals
        _case("sal", 8_000_000, 0, name="sal_8m"),
        # a serving moment: requests of very different sizes on one context
        _case("serve", 60_000, 250, host=True, name="serve_60k"),
    ]


def draw(rng):
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["reads", "reads", "reads", "host", "plain", "long", "seeds", "smem", "sal", "serve"])
    if kind == "reads":
        return _case("reads", size(64, 2_000_000), rng.randint(76, 250),
                     n_rate=rng.choice([0.0, 0.0, 0.0, 0.001, 0.003]), match=rng.choice([1, 1, 1, 2]))
    if kind == "host":
        return _case("reads", size(64, 1_000_000), rng.randint(76, 250), host=True,
                     n_rate=rng.choice([0.0, 0.0, 0.001]))
    if kind == "plain":
        return _case("plain", size(64, 200_000), 130)
    if kind == "long":
        rl = size(600, 10_000)
        return _case("long", size(32, min(20_000, 100_000_000 // rl)), rl)
    if kind == "seeds":
        return _case("seeds", size(1000, 100_000), rng.choice([151, 250]), host=True)
    if kind == "smem":
        return _case("smem", size(1000, 200_000), rng.choice([100, 151, 250]), host=True)
    if kind == "sal":
        return _case("sal", size(10_000, 8_000_000), 0)
    return _case("serve", size(2_000, 60_000), rng.choice([151, 250]), host=True)


# ------------------------------------------------------------------ what a mapper keeps

def _params(case):
    a = case["match"]
    sc = workload.Scoring(a, 4 * a, 6 * a, a, 6 * a, a)
    if case["kind"] == "long":
        return workload.Params(sc, w=500, zdrop=400 * a, end_bonus=5 * a)
    return workload.Params(sc, w=100, zdrop=100 * a, end_bonus=5 * a)


@functools.lru_cache(maxsize=None)
def _context(params, long_queries, what):
    """One context per parameter set; what: 'extend', 'seeds', 'smem', 'sal' or 'serve', with its index loaded."""
    ctx = bsw.Context(params, BUDGET)
    if long_queries:
        ctx.set_plan(bsw.make_plan(short_max=128, warp_x2=1))
    if what == "seeds":
        ctx.set_reference(workload.reference())
    elif what == "smem":
        ctx.fm_build(workload.reference()[:FM_BASES])
    elif what == "sal":
        # the lookup only moves the entries, so any permutation stands for the suffix array
        ctx.sal_set_index(_suffix_array().cpu().numpy())
    return ctx


def _ctx(case):
    what = case["kind"] if case["kind"] in ("seeds", "smem", "sal", "serve") else "extend"
    return _context(_params(case), case["kind"] == "long", what)


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


@functools.lru_cache(maxsize=None)
def _reference():
    return torch.randint(0, 4, (REF_BASES,), dtype=torch.uint8, device="cuda", generator=_gen(1))


@functools.lru_cache(maxsize=None)
def _suffix_array():
    return torch.randperm(SA_ENTRIES, dtype=torch.int32, device="cuda", generator=_gen(2))


# ------------------------------------------------------------------ extension pairs

def _lengths(case, n, g):
    """Query lengths and seed scores of n pairs."""
    dev = "cuda"
    if case["kind"] == "plain":
        return (torch.randint(1, 131, (n,), device=dev, generator=g),
                torch.randint(19, 61, (n,), device=dev, generator=g) * case["match"])
    if case["kind"] == "long":
        u = torch.rand(n, device=dev, dtype=torch.float64, generator=g)
        ql = torch.exp(u * math.log(case["read_len"])).round().long().clamp(1, case["read_len"])
        return ql, torch.randint(19, 61, (n,), device=dev, generator=g) * case["match"]
    reads, rl = (n + 1) // 2, case["read_len"]
    seed = (19 + torch.rand(reads, device=dev, generator=g) * (rl - 18)).long().clamp(max=rl)
    left = (torch.rand(reads, device=dev, generator=g) * (rl - seed + 1)).long()
    left = torch.minimum(left, rl - seed)
    ql = torch.stack([left, rl - seed - left], 1).reshape(-1)[:n]
    return ql, torch.repeat_interleave(seed * case["match"], 2)[:n]


def _dense(case, ql, g):
    """Codes of queries and targets as rows, 0 past their ends, and masks of the N bases (None without N)."""
    p, n, dev, ref = _params(case), ql.shape[0], "cuda", _reference()
    wq = (int(ql.max()) + 15) // 16 * 16 if n else 16
    wq = max(wq, 16)
    wt = (wq + p.w + 15) // 16 * 16
    start = torch.randint(0, REF_BASES - 2 * wt - 64, (n, 1), device=dev, generator=g)
    sub, indel, most = {"plain": (0.01, 0.001, 3), "long": (0.06, 0.03, 3)}.get(
        case["kind"], (0.011, 0.0, 1) if case["read_len"] == 151 else (0.018, 0.0011, 10))
    j = torch.arange(wt, device=dev)
    tl = (ql + p.w)[:, None]
    t = torch.where(j < tl, ref[start + j], 0).to(torch.uint8)
    jq = j[:wq]
    pos = start + jq
    ins = None
    if indel:
        hit = torch.rand(n, wq, device=dev, generator=g)
        size = torch.randint(1, most + 1, (n, wq), device=dev, generator=g, dtype=torch.int16)
        begin = hit < indel / 2
        ins = begin.clone()
        for k in range(1, most):
            ins[:, k:] |= begin[:, :-k] & (size[:, :-k] > k)
        step = torch.where((hit >= indel / 2) & (hit < indel), size, 0) - ins.to(torch.int16)
        pos = (pos + torch.cumsum(step, 1)).clamp_(0, REF_BASES - 1)
        del hit, size, begin, step
    q = ref[pos]
    u = torch.rand(n, wq, device=dev, generator=g)
    other = torch.randint(1, 4, (n, wq), device=dev, generator=g, dtype=torch.uint8)
    q = torch.where((u < sub), (q + other) & 3, q)
    if ins is not None:
        q = torch.where(ins, other ^ (u < 0.5).to(torch.uint8), q)
    q = torch.where(jq < ql[:, None], q, 0).to(torch.uint8)
    if not case["n_rate"]:
        return q, t, None, None
    qn = (torch.rand(n, wq, device=dev, generator=g) < case["n_rate"]) & (jq < ql[:, None])
    run = torch.randint(1, 41, (n, wt), device=dev, generator=g, dtype=torch.int16)
    run = torch.where(torch.rand(n, wt, device=dev, generator=g) < 0.2 * case["n_rate"], run + j.to(torch.int16), 0)
    tn = (torch.cummax(run, 1).values > j) & (j < tl)
    return q.masked_fill(qn, 0), t.masked_fill(tn, 0), qn, tn


def _chunks(case, seed):
    """The pairs of a case in chunks: (query lengths, scores, q rows, t rows, q N rows, t N rows)."""
    g = _gen(seed)
    ql, h0 = _lengths(case, case["n"], g)
    wide = case["read_len"] + _params(case).w + 32
    rows = max(1, (1 << 26) // wide)
    for s in range(0, case["n"], rows):
        yield (ql[s:s + rows], h0[s:s + rows], *_dense(case, ql[s:s + rows], g))


def _packed(rows, lens, per):
    """Rows of codes (per 4: four 2-bit codes a byte) or bits (per 8) as bytes, each row cut at a multiple of 16."""
    w = torch.tensor([1 << (8 // per * k) for k in range(per)], dtype=torch.uint8, device="cuda")
    b = (rows.to(torch.uint8).view(rows.shape[0], -1, per) * w).sum(2, dtype=torch.uint8)
    return b[torch.arange(b.shape[1], device="cuda") < ((lens + 15) // 16 * (16 // per))[:, None]]


class Pairs:
    """A packed batch with its result buffers, in device memory or, for the calls on host buffers, pinned."""

    def __init__(self, case, seed):
        parts = [[] for _ in range(6)]
        for ql, h0, q, t, qn, tn in _chunks(case, seed):
            tl = ql + _params(case).w
            for part, v in zip(parts, (ql, h0, _packed(q, ql, 4), _packed(t, tl, 4),
                                       None if qn is None else _packed(qn, ql, 8),
                                       None if tn is None else _packed(tn, tl, 8))):
                part.append(v)
        ql, h0, q, t, qn, tn = (None if p[0] is None else torch.cat(p) for p in parts)
        tl = ql + _params(case).w

        def place(x):
            return x.cpu().pin_memory() if case["host"] else x

        def offsets(n):
            n = (n + 15) // 16 * 16
            return place(torch.cumsum(n, 0) - n)

        pad = torch.zeros(16, dtype=torch.uint8, device="cuda")
        self.n, self.flags, self.host = int(ql.shape[0]), 0, case["host"]
        self.q, self.t = place(torch.cat([q, pad])), place(torch.cat([t, pad]))
        self.q_n, self.t_n = (None if x is None else place(torch.cat([x, pad])) for x in (qn, tn))
        self.q_off, self.t_off = offsets(ql), offsets(tl)
        self.q_len, self.t_len, self.h0 = (place(x.to(torch.int32)) for x in (ql, tl, h0))
        self.out = torch.zeros((self.n, 6), dtype=torch.int32, device="cpu" if self.host else "cuda",
                               pin_memory=self.host)
        self.cells = torch.zeros(1, dtype=torch.int64, device="cuda")

    def struct(self, flags=0):
        return bsw.bsw_batch_t(self.n, self.q.data_ptr(), self.q_off.data_ptr(), self.q_len.data_ptr(),
                               self.t.data_ptr(), self.t_off.data_ptr(), self.t_len.data_ptr(), self.h0.data_ptr(),
                               None, flags | (0 if self.host else bsw.BSW_DEVICE_PTRS),
                               None if self.q_n is None else self.q_n.data_ptr(),
                               None if self.t_n is None else self.t_n.data_ptr())


def _request_sizes(total):
    """Sizes of a burst of requests: a few large, most small."""
    sizes = []
    while total > 0 and len(sizes) < 23:
        sizes.append((total + 2) // 3 if len(sizes) % 2 == 0 else total // 17 + 1)
        total -= sizes[-1]
    return sizes + [total] if total else sizes


# ------------------------------------------------------------------ the cases' calls

def prepare(case, seed):
    kind, ctx = case["kind"], _ctx(case)
    state = {"kind": kind, "ctx": ctx, "host": case["host"]}
    if kind in ("reads", "plain", "long"):
        state["batch"] = Pairs(case, seed)
    elif kind == "serve":
        state["batches"] = [Pairs(dict(case, kind="reads", n=s, read_len=151 if k % 3 == 2 else case["read_len"]),
                                  seed * 64 + k) for k, s in enumerate(_request_sizes(case["n"]))]
    elif kind == "seeds":
        name = "seeds151" if case["read_len"] == 151 else "seeds250"
        state["prep"] = ctx.prepare_seeds(workload.make_seeds(name, case["n"], seed=seed))
        state["out"] = np.zeros(2 * case["n"], bsw.ALN_DTYPE)
    elif kind == "smem":
        codes, off, length, _ = workload.make_reads(case["n"], case["read_len"], FM_BASES, seed=seed)
        state["reads"] = (bsw.bsw_pack_2bit(codes), off, length)
        state["out"] = np.zeros(4 * case["n"] + 16, bsw.SMEM_DTYPE)
        state["first"] = np.zeros(case["n"] + 1, np.int64)
        state["found"] = np.zeros(1, np.int64)
    elif kind == "sal":
        state["intervals"] = _intervals(case, seed)
        state["out"] = torch.zeros(_positions_room(case), dtype=torch.int32, device="cuda")
    return state


def _intervals(case, seed):
    """Suffix array intervals at random rows, a quarter of them of one hit, the rest geometric (at most 500)."""
    g, n = _gen(seed), case["n"]
    u = torch.rand(n, device="cuda", dtype=torch.float64, generator=g)
    cnt = (1 + (torch.log1p(-u) / math.log(0.75)).long()).clamp(1, 500)
    k = (torch.rand(n, device="cuda", dtype=torch.float64, generator=g) * (SA_ENTRIES - 500)).long()
    return k, cnt.to(torch.int32), torch.cumsum(cnt, 0) - cnt


def _positions_room(case):
    """Room for the positions of any case["n"] intervals: four each, and nine standard deviations."""
    return 4 * case["n"] + 32 * math.isqrt(case["n"]) + 500


def run(state):
    kind, ctx = state["kind"], state["ctx"]
    if kind in ("reads", "plain", "long"):
        b = state["batch"]
        if state["host"]:
            out, cells = ctx.extend_host(b, out=b.out.numpy())
            return {"out": out, "cells": cells}
        ctx.extend_device(b)
        return {"out": b.out, "cells": b.cells}
    if kind == "serve":
        tickets = [ctx.submit(b, b.out.numpy()) for b in state["batches"]]
        for t in tickets:
            if ctx.poll(t) != bsw.BSW_OK:
                raise RuntimeError("a request failed")
        return [b.out for b in state["batches"]]
    if kind == "seeds":
        out, cells = ctx.extend_prepared(state["prep"], out=state["out"])
        return {**{f: out[f] for f in bsw.ALN_DTYPE.names}, "cells": cells}
    if kind == "smem":
        reads, off, length = state["reads"]
        out, first, found = state["out"], state["first"], state["found"]
        rc = bsw.lib().bsw_smem(ctx.handle, length.shape[0], reads.ctypes.data, off.ctypes.data, length.ctypes.data, 19,
                                out.ctypes.data, out.shape[0], found.ctypes.data, first.ctypes.data)
        if rc != bsw.BSW_OK:
            raise bsw.BswError(rc, "bsw_smem")
        return {**{f: out[f] for f in ("read_id", "qbeg", "len", "k", "s")}, "first": first, "found": found}
    ctx.sal_lookup_device(*state["intervals"], state["out"])
    return state["out"]


# ------------------------------------------------------------------ what a pass cannot do without

def _mean_query(case):
    if case["kind"] == "plain":
        return 65.5
    if case["kind"] == "long":
        return case["read_len"] / math.log(case["read_len"])
    return (case["read_len"] - 19) / 4


def _pair_work(n, q, w, cells, n_bits):
    seq = (q + q + w) / 4 * (1.5 if n_bits else 1.0)
    # offsets, lengths and h0 in, six fields out; seven integer operations a cell
    return {"bytes": n * (seq + 28 + 24), "flops": 7.0 * n * cells}


def work(case):
    kind, n, rl = case["kind"], case["n"], case["read_len"]
    q = _mean_query(case)
    # cells inside the trimmed band, per pair, as measured on the benchmark's batches
    cells = {"plain": 6580.0, "long": 676.0 * q}.get(kind, 0.108 * rl * rl)
    if kind in ("reads", "plain", "long", "serve"):
        return _pair_work(n, q, 500 if kind == "long" else 100, cells, case["n_rate"] > 0)
    if kind == "seeds":
        w = _pair_work(4 * n, (rl - 35) / 2, 100, 0.245 * rl * rl, False)
        return {"bytes": w["bytes"] + 2 * n * 72.0, "flops": w["flops"]}
    if kind == "smem":
        # the reads in, about two records a read out; two table entries and some twenty operations for each base
        # taken, forward and back
        return {"bytes": n * (rl / 4 + 12 + 2 * 40 + 8.0), "flops": n * 2.0 * rl * 20}
    return {"bytes": n * (20 + 4 * 8.0), "flops": 0.0}


def tolerance(case):
    return "exact"


# ------------------------------------------------------------------ the same in 64-bit torch

def exact(case, seed):
    if case["kind"] == "sal":
        k, cnt, off = _intervals(case, seed)
        c = cnt.long()
        i = torch.arange(int(c.sum()), device="cuda") - torch.repeat_interleave(off, c)
        out = torch.zeros(_positions_room(case), dtype=torch.int64, device="cuda")
        out[:i.shape[0]] = _suffix_array()[torch.repeat_interleave(k, c) + i]
        return out
    if case["kind"] not in ("reads", "plain") or case["n"] > 20_000:
        return None
    outs, cells = [], 0
    for ql, h0, q, t, qn, tn in _chunks(case, seed):
        o, c = _extend(_params(case), ql, h0.long(), q, t, qn, tn)
        outs.append(o)
        cells += c
    out = torch.cat(outs)
    return {"out": out.cpu().numpy() if case["host"] else out,
            "cells": cells if case["host"] else torch.tensor([cells], device="cuda")}


def _extend(p, n, h0, q, t, qn, tn):
    """BWA-MEM's extension (affine gaps, band, z-drop, trimmed ends) of all pairs, a row of every pair at a time."""
    s, m = p.scoring, n + p.w
    neg = -(1 << 40)
    oe_d, oe_i = s.o_del + s.e_del, s.o_ins + s.e_ins

    def cap(o, e):
        return ((n * s.match + p.end_bonus - o + e).div(e, rounding_mode="trunc")).clamp(min=1)

    wb = torch.minimum(cap(s.o_ins, s.e_ins), cap(s.o_del, s.e_del)).clamp(max=p.w)[:, None]
    cols = torch.arange(q.shape[1] + 1, device="cuda")[None, :]
    n1, h1 = n[:, None], h0[:, None]
    H = torch.where(cols == 0, h1, (h1 - s.o_ins - cols * s.e_ins).clamp(min=0))
    H = torch.where(cols <= n1, H, 0)
    E = torch.zeros_like(H)
    q = torch.nn.functional.pad(q.long(), (0, 1))
    lo, hi = torch.zeros_like(n1), n1.clone()
    best, bi, bj = h1.clone(), torch.full_like(n1, -1), torch.full_like(n1, -1)
    gbest, gi, moff = torch.full_like(n1, -1), torch.full_like(n1, -1), torch.zeros_like(n1)
    live, cells = n1 > 0, 0
    for i in range(int(m.max()) if n.numel() else 0):
        live = live & (i < m[:, None])
        if not bool(live.any()):
            break
        lo = torch.where(live, torch.maximum(lo, i - wb), lo)
        hi = torch.where(live, torch.minimum(torch.minimum(hi, i + wb + 1), n1), hi)
        on = live & (cols >= lo) & (cols < hi)
        cells += int(on.sum())
        left = torch.where(lo == 0, (h1 - s.o_del - (i + 1) * s.e_del).clamp(min=0), 0)
        sc = torch.where(q == t[:, i:i + 1].long(), s.match, -s.mismatch)
        if qn is not None:
            sc = torch.where(torch.nn.functional.pad(qn, (0, 1)) | tn[:, i:i + 1], -1, sc)
        M = torch.where(H > 0, H + sc, 0)
        # F(j) = max over k < j of M(k) - o - (j - k) e, at least 0
        run = torch.cummax(torch.where(on, M - oe_i + (cols + 1) * s.e_ins, neg), 1).values
        F = (torch.nn.functional.pad(run, (1, 0), value=neg)[:, :-1] - cols * s.e_ins).clamp(min=0)
        h = torch.where(on, torch.maximum(torch.maximum(M, E), F), 0)
        E2 = torch.maximum(E - s.e_del, M - oe_d).clamp(min=0)
        rm = h.max(1, keepdim=True).values
        rj = torch.where(on & (h == rm), cols, -1).max(1, keepdim=True).values
        prev = torch.nn.functional.pad(h, (1, 0))[:, :-1]
        prev = torch.where(cols == lo, left, prev)
        last = torch.where(hi > lo, h.gather(1, (hi - 1).clamp(min=0)), left)
        H = torch.where(on, prev, H)
        E = torch.where(on, E2, E)
        at_end = live & (cols == hi)
        H = torch.where(at_end, last, H)
        E = torch.where(at_end, 0, E)
        full = live & (torch.maximum(lo, hi) == n1)
        gi = torch.where(full & (last >= gbest), i, gi)
        gbest = torch.where(full, torch.maximum(gbest, last), gbest)
        up = live & (rm > best)
        di, dj = i - bi, rj - bj
        drop = best - rm - torch.where(di > dj, (di - dj) * s.e_del, (dj - di) * s.e_ins)
        stop = (rm == 0) | (~up & (p.zdrop > 0) & (drop > p.zdrop))
        best, bi, bj = torch.where(up, rm, best), torch.where(up, i, bi), torch.where(up, rj, bj)
        moff = torch.where(up, torch.maximum(moff, (rj - i).abs()), moff)
        live = live & ~stop
        some = (H != 0) | (E != 0)
        lo2 = torch.where(some & (cols >= lo) & (cols < hi), cols, hi).min(1, keepdim=True).values
        end = torch.where(some & (cols >= lo2) & (cols <= hi), cols, lo2 - 1).max(1, keepdim=True).values
        lo, hi = torch.where(live, lo2, lo), torch.where(live, torch.minimum(end + 2, n1), hi)
    gbest = torch.where(n1 == 0, h1, gbest)
    return torch.cat([best, bj + 1, bi + 1, gi + 1, gbest, moff], 1), cells
