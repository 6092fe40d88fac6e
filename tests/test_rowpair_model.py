"""The row-pair scheme against the oracle, on the host (no GPU).

`rowpair_model.extend` restates the kernels' two-rows-per-instruction pass bit
by bit (packed instructions emulated on 32-bit words), for the 8-bit lanes
without and with N bases and for the 16-bit lanes.  These tests pin the scheme
itself: every result field and the cell count equal the oracle's for random
pairs under symmetric and split gap costs, match scores 1 to 3 and bands of 0
to 100 columns (16-bit lanes: match scores up to 127 and bounds up to 2047);
for pairs whose rows read slots past the previous row's end (the oracle counts
those reads); and for every row count from 1 to 9.  The GPU tests in
`test_gpu_rowpair.py`, `test_gpu_nbase.py` and `test_gpu_rows16.py` check the
kernels on the same kinds of input.
"""
import numpy as np
import pytest

import oracle
import rowpair_model
from paper_1907_12931_gb300 import workload as W


def random_case(rng):
    a = int(rng.integers(1, 4))
    b = int(rng.integers(1, 6))
    od, ed = int(rng.integers(0, 8)), int(rng.integers(1, 3))
    oi, ei = (od, ed) if rng.random() < 0.5 else (int(rng.integers(0, 8)), int(rng.integers(1, 3)))
    n, m = int(rng.integers(1, 61)), int(rng.integers(1, 91))
    ref = rng.integers(0, 4, n + m + 10)
    q = ref[:n].copy()
    flip = rng.random(n) < rng.choice([0.0, 0.02, 0.1, 0.4])
    q[flip] = rng.integers(0, 4, int(flip.sum()))
    off = int(rng.integers(0, 6))
    t = ref[off:off + m].copy() if rng.random() < 0.7 else rng.integers(0, 4, m)
    left = 255 - a * min(n, m)
    h0 = int(rng.integers(0, min(left, 120) + 1)) if left >= 0 else None
    params = W.Params(W.Scoring(a, b, od, ed, oi, ei), w=int(rng.choice([0, 1, 2, 3, 5, 10, 30, 100])),
                      zdrop=int(rng.choice([0, 1, 5, 20, 100])), end_bonus=int(rng.integers(0, 8)))
    return params, q.astype(np.uint8), t.astype(np.uint8), h0


def same(params, q, t, h0, what, lanes=({}, {"nm": True}, {"lane": rowpair_model.Lane16})):
    """On each lane: 8-bit without N codes and with them (none in the pair), 16-bit."""
    ref, cells, stale = oracle.extend_one(params, q, t, h0)
    for lane in lanes:
        got, gc = rowpair_model.extend(params, q, t, h0, **lane)
        assert got == ref and gc == cells, (what, lane, len(q), len(t), h0, params, ref, cells, got, gc)
    return stale


@pytest.mark.parametrize("seed", range(4))
def test_random_pairs(seed):
    rng = np.random.default_rng(900 + seed)
    done = 0
    while done < 400:
        params, q, t, h0 = random_case(rng)
        if h0 is None:
            continue
        same(params, q, t, h0, "random %d" % seed)
        done += 1


def test_stale_slot_reads():
    """Narrow bands and large h0 over near copies: rows whose band end grows
    by two columns read slots an earlier row wrote."""
    rng = np.random.default_rng(77)
    with_stale = tries = 0
    while with_stale < 60 and tries < 60000:
        tries += 1
        a = int(rng.integers(1, 4))
        n, m = int(rng.integers(2, 50)), int(rng.integers(2, 60))
        q = rng.integers(0, 4, n).astype(np.uint8)
        t = (q[rng.integers(0, n, m)] if rng.random() < 0.5 else rng.integers(0, 4, m)).astype(np.uint8)
        left = 255 - a * min(n, m)
        if left < 0:
            continue
        h0 = int(rng.integers(0, min(left, 80) + 1))
        od, ed = int(rng.integers(0, 6)), int(rng.integers(1, 3))
        params = W.Params(W.Scoring(a, int(rng.integers(1, 6)), od, ed, od, ed),
                          w=int(rng.choice([1, 2, 3, 5, 8])), zdrop=int(rng.choice([0, 3, 30])),
                          end_bonus=int(rng.integers(0, 6)))
        ref, cells, stale = oracle.extend_one(params, q, t, h0)
        if stale == 0:
            continue
        with_stale += 1
        same(params, q, t, h0, "stale")
    assert with_stale >= 60, with_stale


def test_row_counts():
    """Target lengths 1 to 9 (the last row alone when odd) against queries
    of 1 to 12 bases."""
    rng = np.random.default_rng(3)
    for m in range(1, 10):
        for n in range(1, 13):
            for h0 in (0, 1, 7, 30, 200):
                if h0 + min(n, m) > 255:
                    continue
                q = rng.integers(0, 4, n).astype(np.uint8)
                t = np.where(rng.random(m) < 0.8, np.resize(q, m), rng.integers(0, 4, m)).astype(np.uint8)
                for w in (0, 1, 2, 100):
                    same(W.Params(W.Scoring(), w=w, zdrop=1, end_bonus=5), q, t, h0, "rows")


@pytest.mark.parametrize("seed", range(2))
def test_n_bases(seed):
    """N in queries and targets, on the 8-bit lane that takes them."""
    rng = np.random.default_rng(950 + seed)
    done = 0
    while done < 200:
        params, q, t, h0 = random_case(rng)
        if h0 is None:
            continue
        q[rng.random(len(q)) < rng.choice([0.0, 0.02, 0.3])] = 4
        t[rng.random(len(t)) < rng.choice([0.0, 0.02, 0.3])] = 4
        same(params, q, t, h0, "N %d" % seed, lanes=({"nm": True},))
        done += 1


@pytest.mark.parametrize("seed", range(4))
def test_scores_past_eight_bits(seed):
    """The 16-bit lane at bounds from 256 to 2047, under match scores up to 127
    and gap costs past the largest score."""
    rng = np.random.default_rng(970 + seed)
    done = 0
    while done < 150:
        a = int(rng.choice([1, 2, 5, 20, 60, 127]))
        n, m = int(rng.integers(1, 61)), int(rng.integers(1, 91))
        left = 2047 - a * min(n, m)
        if left < 0:
            continue
        h0 = left if done % 3 == 0 else int(rng.integers(0, left + 1))
        q = rng.integers(0, 4, n).astype(np.uint8)
        t = np.where(rng.random(m) < 0.9, np.resize(q, m), rng.integers(0, 4, m)).astype(np.uint8)
        od, ed = int(rng.choice([0, 6, 200, 3000])), int(rng.choice([1, 2, 40]))
        oi, ei = (od, ed) if rng.random() < 0.5 else (int(rng.choice([0, 9, 2500])), int(rng.choice([1, 7])))
        params = W.Params(W.Scoring(a, int(rng.choice([1, 4, 40, 128])), od, ed, oi, ei),
                          w=int(rng.choice([0, 1, 3, 10, 100])), zdrop=int(rng.choice([0, 20, 500])), end_bonus=5)
        same(params, q, t, h0, "bound %d" % (2047 - left + h0), lanes=({"lane": rowpair_model.Lane16},))
        done += 1


def test_packed_helpers():
    """The emulated packed instructions act on each 16-bit half alone."""
    m = rowpair_model
    for lo_a, hi_a, lo_b, hi_b, lo_c, hi_c in [(5, -3, 2, 7, 4, -9), (-100, 200, 50, -50, 0, 0), (255, 0, 3, -4, 256, 1)]:
        a, b, c = m.pack(lo_a, hi_a), m.pack(lo_b, hi_b), m.pack(lo_c, hi_c)
        assert m.viaddmin_s16x2(a, b, c) == m.pack(min(lo_a + lo_b, lo_c), min(hi_a + hi_b, hi_c))
        assert m.viaddmax_s16x2(a, b, c) == m.pack(max(lo_a + lo_b, lo_c), max(hi_a + hi_b, hi_c))
        assert m.vimax3_s16x2(a, b, c) == m.pack(max(lo_a, lo_b, lo_c), max(hi_a, hi_b, hi_c))
        assert m.sub_sat_h2(a, m.pack(7, 11)) == m.pack(max(0, lo_a - 7), max(0, hi_a - 11))
    # the selector of slot j gives s(t_i, q_j) high and s(t_{i+1}, q_{j-1}) low, sign-extended
    params = W.Params(W.Scoring(1, 4, 6, 1, 6, 1))
    for nm in (False, True):
        for qj in range(5 if nm else 4):
            for qjm in range(5 if nm else 4):
                lane = m.Lane8(params.scoring, [qjm, qj], 0, nm)
                lane.rows(3, 1)
                r = lane.scores(lane.S[1])
                assert m.hi16(r) == (-1 if qj == 4 else 1 if qj == 3 else -4)
                assert m.lo16(r) == (-1 if qjm == 4 else 1 if qjm == 1 else -4)
                assert lane.score0(1) == m.hi16(r)
                assert lane.score1(0) == m.lo16(r)
