"""The 16-bit per-thread kernel's row pairs against the oracle (needs a GPU).

Pairs of the 16-bit classes up to a score bound of 2047 run two rows per
packed instruction, the others one row at a time.  The cases sit at that line
(h0 + match * min(n, m) at 2046 to 2049), at the code words' and blocks' edges
(query lengths around multiples of 8, and each class's bound), and at row
counts of one to nine.  Every comparison is bit-exact on all six result fields
and the cell count.  A batch with bounds on both sides of the line costs no more
than one with all of them past it.
"""
import time

import numpy as np
import pytest

import oracle
from paper_1907_12931_gb300 import workload as W
from test_gpu_parity import NTH, assert_same, run

pytestmark = pytest.mark.gpu

LENGTHS = [1, 2, 7, 8, 9, 15, 16, 17, 31, 32, 33, 63, 64, 65, 127, 128, 129, 247, 248, 255, 256]


@pytest.fixture(scope="module")
def bsw():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1907_12931_gb300 import bsw as _b
    _b.lib()
    return _b


def near_copy(rng, n, m):
    ref = rng.integers(0, 4, n + m + 8)
    q = ref[:n].copy()
    flip = rng.random(n) < rng.choice([0.0, 0.03, 0.3])
    q[flip] = rng.integers(0, 4, int(flip.sum()))
    off = int(rng.integers(0, 4))
    t = ref[off:off + m] if rng.random() < 0.8 else rng.integers(0, 4, m)
    return q.astype(np.uint8), t.astype(np.uint8)


@pytest.mark.parametrize("sc,w,zd", [((1, 4, 6, 1, 6, 1), 100, 100), ((2, 8, 12, 2, 12, 2), 100, 200),
                                     ((3, 5, 4, 2, 7, 1), 9, 0), ((7, 9, 3000, 40, 2000, 50), 40, 60)])
def test_edges(bsw, sc, w, zd):
    rng = np.random.default_rng(sc[0] * 100 + w)
    qs, ts, hs = [], [], []
    for n in LENGTHS:
        for m in list(range(1, 10)) + [n + 1, n + 30, n + 101]:
            q, t = near_copy(rng, n, m)
            top = sc[0] * min(n, m)
            for bound in (2046, 2047, 2048, 2049, top, top + 40, top + 300):
                if bound >= top:
                    qs.append(q); ts.append(t); hs.append(bound - top)
    wl = W.from_lists(qs, ts, hs, W.Params(W.Scoring(*sc), w=w, zdrop=zd, end_bonus=5), align=4)
    ref, cells, _ = oracle.extend_batch(wl, nthreads=NTH)
    for flags in (0, bsw.BSW_FORCE_I16):
        got, gc = run(bsw, wl, flags=flags, device=True)
        assert_same(got, ref, "16-bit rows %s w=%d flags %d" % (sc, w, flags))
        assert gc == int(cells.sum())


@pytest.mark.parametrize("bounds", [0xf, 0x1, 0x5])
def test_bounds_on_both_sides(bsw, bounds):
    """Every second pair past the line, in all classes and with classes of
    several lengths merged: no warp runs both ways, so the batch takes less than
    one of the slower kind alone (half a kind each: about 0.75 of it; in warps
    that mix them 1.4)."""
    rng = np.random.default_rng(bounds)
    m1 = 4096
    qs, ts = zip(*[near_copy(rng, int(n), int(n) + 60) for n in rng.choice([30, 60, 120, 121, 250], m1)])
    k = np.arange(160_000)
    params = W.Params(W.Scoring(8, 32, 48, 8, 48, 8), w=100, zdrop=800, end_bonus=40)
    ms = {}
    for name, past in (("both", k % 2 == 0), ("past", k >= 0)):
        hs = [int((2100 if p else 2047) - 8 * len(qs[j % m1])) for j, p in zip(k, past)]
        assert min(hs) >= 0
        wl = W.from_lists([qs[j % m1] for j in k], [ts[j % m1] for j in k], hs, params, align=4)
        if name == "both":
            ref, cells, _ = oracle.extend_batch(wl, nthreads=NTH)
        with bsw.Context(params, 4 << 30) as ctx:
            ctx.set_plan(bsw.make_plan(i16_bounds=bounds))
            db = bsw.DeviceBatch(bsw.HostBatch(wl))
            t = []
            for _ in range(8):
                ctx.sync()
                t0 = time.perf_counter()
                ctx.extend_device(db)
                ctx.sync()
                t.append(1e3 * (time.perf_counter() - t0))
            if name == "both":
                assert_same(db.out.cpu().numpy(), ref, "both sides, bounds %x" % bounds)
                assert int(db.cells.item()) == int(cells.sum())
        ms[name] = min(t[2:])
    assert ms["both"] < ms["past"], ms
