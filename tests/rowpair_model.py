"""A bit-level model of the row-pair pass, for CPU tests.

The per-thread kernels run rows i and i+1 of a pair in the high and low halves
of 32-bit registers, row i+1 one column behind, and settle row i+1's band ends
from row i after the fact (the kernel's comment gives the argument).  This
module restates that pass in Python with every packed instruction emulated on
32-bit words: DPX add-min / add-max / three-way max per 16-bit half, byte
permutes, multiplies that wrap at 32 bits, funnel shifts, and the
half-precision subtraction and product with .sat on the halves' bit patterns.
The slot column is a list of 32-bit words in the kernel's layout.  Lane8 is the
8-bit lane, with and without N bases, Lane16 the 16-bit lane with its code
words and block keys; both take steps in blocks of 8, 4, 2 and 1 as the kernel
does, all of a block's slots read before the first is written back.

`tests/test_rowpair_model.py` checks the pass against the oracle on the host:
the band start found before the packed loop, the band end from the last
positive column of row i, row i's zeros written back past row i+1's end, reads
of slots past the previous row's end (the band rule of Section V-A), the last
row alone when the row count is odd.

It is test infrastructure: nothing outside `tests/` imports it, and it shares
no code with the CUDA path or the oracle (it calls the oracle only for the
clipped band width w').
"""
import functools

import numpy as np

import oracle

M32 = 0xffffffff


def s16(x):
    x &= 0xffff
    return x - 0x10000 if x & 0x8000 else x


def lo16(x):
    return s16(x)


def hi16(x):
    return s16(x >> 16)


def pack(lo, hi):
    return (lo & 0xffff) | ((hi & 0xffff) << 16)


def u16lo(x):
    return x & 0xffff


def u16hi(x):
    return (x >> 16) & 0xffff


# Per-half emulations of the DPX instructions the kernels use.
def viaddmin_s16x2(a, b, c):
    return pack(min(s16(lo16(a) + lo16(b)), lo16(c)), min(s16(hi16(a) + hi16(b)), hi16(c)))


def viaddmax_s16x2(a, b, c):
    return pack(max(s16(lo16(a) + lo16(b)), lo16(c)), max(s16(hi16(a) + hi16(b)), hi16(c)))


def vimax3_s16x2(a, b, c):
    return pack(max(lo16(a), lo16(b), lo16(c)), max(hi16(a), hi16(b), hi16(c)))


def viaddmax_u16x2(a, b, c):
    return pack(max((u16lo(a) + u16lo(b)) & 0xffff, u16lo(c)), max((u16hi(a) + u16hi(b)) & 0xffff, u16hi(c)))


def mul(a, b):
    return (a * b) & M32


def funnelshift_r(lo, hi, sh):
    return (((hi << 32) | lo) >> (sh & 31)) & M32


def prmt(a, b, sel):
    """Byte permute: output byte k is byte (nibble k & 7) of {a, b}, or that
    byte's sign replicated when the nibble's bit 3 is set."""
    by = [(a >> (8 * k)) & 0xff for k in range(4)] + [(b >> (8 * k)) & 0xff for k in range(4)]
    out = 0
    for k in range(4):
        nib = (sel >> (4 * k)) & 0xf
        v = by[nib & 7]
        if nib & 8:
            v = 0xff if v & 0x80 else 0
        out |= v << (8 * k)
    return out


# Half precision on bit patterns: the exact result, rounded to nearest even,
# clamped to [0, 1] with NaN as +0 (.sat).  A double holds any difference or
# product of two halves exactly.
def _half(bits):
    return float(np.uint16(bits).view(np.float16))


def _sat_bits(x):
    x = 0.0 if x != x else min(max(x, 0.0), 1.0)
    return int((np.float16(x) + np.float16(0.0)).view(np.uint16))


@functools.lru_cache(maxsize=None)
def sub_sat_h(a, b):
    return _sat_bits(_half(a) - _half(b))


@functools.lru_cache(maxsize=None)
def mul_sat_h(a, b):
    return _sat_bits(_half(a) * _half(b))


def sub_sat_h2(a, b):
    return sub_sat_h(a & 0xffff, b & 0xffff) | sub_sat_h(a >> 16, b >> 16) << 16


def positive_h2(x):
    return mul_sat_h(x & 0xffff, 0x7c00) | mul_sat_h(x >> 16, 0x7c00) << 16


def sext8(x):
    x &= 0xff
    return x - 256 if x & 0x80 else x


N_SCORE = 0xffffffff                           # -1 in every byte: an N against anything


class Row:
    """Running values of a row-pair pass: high halves row i, low halves row i+1."""

    def __init__(self, hA, hB, EN, F, L):
        self.hA, self.hB, self.EN, self.F, self.L = hA, hB, EN, F, L

    def settle(self, s, hh):
        """The last column of row i with H > 0, plus 1, after steps s.. gave hh."""
        if hh[-1] > 0xffff:
            self.L = s + len(hh)
        else:
            for k in range(len(hh) - 1):
                if hh[k] > 0xffff:
                    self.L = s + k + 1


class Lane:
    """What both lanes share: the scores of the two rows by query code, the gap
    costs in both halves (opening costs clamped at `top`)."""

    def __init__(self, sc, top):
        self.sc = sc
        self.sym = (sc.o_del, sc.e_del) == (sc.o_ins, sc.e_ins)
        self.oe_d2 = min(sc.o_del + sc.e_del, top) * 0x10001
        self.oe_i2 = min(sc.o_ins + sc.e_ins, top) * 0x10001
        self.ne_d2 = (-sc.e_del & 0xffff) * 0x10001
        self.ne_i2 = (-sc.e_ins & 0xffff) * 0x10001

    def rows(self, t0, t1):
        """Target codes of rows i and i+1 (4: N, of a lane that takes N)."""
        mb = -self.sc.mismatch & 0xff
        flip = (self.sc.match ^ mb) & 0xff
        self.p0 = N_SCORE if t0 > 3 else mb * 0x01010101 ^ flip << 8 * t0
        self.p1 = N_SCORE if t1 > 3 else mb * 0x01010101 ^ flip << 8 * t1


class Lane8(Lane):
    """8-bit lanes.  Slot j: the selector in bits 0-15 (nibbles q_{j-1},
    q_{j-1} | 8, 4 + q_j, (4 + q_j) | 8; with N code 4 in the low two, and q_j
    unshifted in the high two), E in 16-23, H in 24-31."""
    KEY = 256

    def __init__(self, sc, q, h0, nm):
        super().__init__(sc, 1023)
        self.nm = nm
        self.S = []
        for j in range(len(q) + 1):
            cj = int(q[j]) if j < len(q) else 0
            cjm = int(q[j - 1]) if j >= 1 else 0
            hv = h0 if j == 0 else max(0, h0 - sc.o_ins - j * sc.e_ins)
            self.S.append(cj * 0x1100 + cjm * 0x11 + (0x8080 if nm else 0xC480) + (hv << 24))

    def put(self, j, h, e):
        self.S[j] = (self.S[j] & 0xffff) | ((((h << 8) | e) & 0xffff) << 16)

    def get(self, j):
        return self.S[j] >> 24, (self.S[j] >> 16) & 0xff

    def nonzero(self, j):
        return self.S[j] >> 16 != 0

    def h_of(self, j):
        return self.S[j] >> 24

    def scores(self, w):
        if not self.nm:
            return prmt(self.p1, self.p0, w)
        return prmt(prmt(self.p1, N_SCORE, w), prmt(self.p0, N_SCORE, w), 0x7610)

    def score0(self, j):
        return hi16(self.scores(self.S[j]))

    def score1(self, j):
        return sext8(prmt(self.p1, N_SCORE, (self.S[j] >> 8) & (7 if self.nm else 3)))

    def open(self, X, c0, bnd1, key_lo):
        X.hK, X.key, X.j2 = bnd1 << 8, key_lo << 16, (c0 + 1) << 16 | c0

    def close(self, X):
        return X.key >> 16, X.key & 0xffff

    def steps(self, s, X, N):
        wv = self.S[s:s + N]
        hh, kb = [], 0
        for k in range(N):
            Hd2 = prmt(X.hB, wv[k], 0x1712)
            Ed2 = prmt(X.EN, wv[k], 0x1612)
            M2 = viaddmin_s16x2(Hd2, self.scores(wv[k]), mul(Hd2, 128))
            h2 = vimax3_s16x2(M2, Ed2, X.F)
            Mi2 = sub_sat_h2(M2, self.oe_i2)
            Md2 = Mi2 if self.sym else sub_sat_h2(M2, self.oe_d2)
            EN2 = viaddmax_s16x2(Ed2, self.ne_d2, Md2)
            X.F = viaddmax_s16x2(X.F, self.ne_i2, Mi2)
            j = s + k - 1
            self.S[j] = (self.S[j] & 0xffff) | ((X.hK + EN2) & 0xffff) << 16
            X.hK = mul(h2, 256)
            kb = X.hK if k == 0 else viaddmax_u16x2(X.hK, k * 0x10001, kb)
            X.hB, X.hA, X.EN = X.hA, h2, EN2
            hh.append(h2)
        X.key = viaddmax_u16x2(kb, X.j2, X.key)
        X.j2 = (X.j2 + N * 0x10001) & M32
        X.settle(s, hh)


class Lane16(Lane):
    """16-bit lanes up to a score bound of 2047.  Slot j: E in the low half, H
    in the high one; the query's codes beside the slots, eight nibbles a word."""
    KEY = 512

    def __init__(self, sc, q, h0, nm):
        assert not nm
        super().__init__(sc, 2047)
        n = len(q)
        self.S = [(h0 if j == 0 else max(0, h0 - sc.o_ins - j * sc.e_ins)) << 16 for j in range(n + 1)]
        # a word past the last column's: a block's codes span two
        self.Q = [sum((int(q[c + k]) if c + k < n else 0) << 4 * k for k in range(8)) for c in range(0, n + 1, 8)] + [0]

    def put(self, j, h, e):
        self.S[j] = h << 16 | e

    def get(self, j):
        return self.S[j] >> 16, self.S[j] & 0xffff

    def nonzero(self, j):
        return self.S[j] != 0

    def h_of(self, j):
        return self.S[j] >> 16

    def score(self, p, j):
        return sext8(prmt(p, 0, (self.Q[j >> 3] >> 4 * (j & 7)) & 3))

    def score0(self, j):
        return self.score(self.p0, j)

    def score1(self, j):
        return self.score(self.p1, j)

    def open(self, X, c0, bnd1, key_lo):
        X.k0, X.k1 = key_lo, 0

    def close(self, X):
        return X.k0, X.k1

    def steps(self, s, X, N):
        w = (s - 1) >> 3
        q0, q1, sh = self.Q[w], self.Q[w + 1], 4 * ((s - 1) & 7)
        cl = funnelshift_r(q0, q1, sh)
        ch = funnelshift_r(cl, q1 >> sh, 4)
        sl = [prmt(self.p1, 0, cl), prmt(self.p1, 0, cl >> 16) if N > 4 else 0]
        sg = [prmt(self.p0, 0, ch), prmt(self.p0, 0, ch >> 16) if N > 4 else 0]
        wv = self.S[s:s + N]
        hh, kb = [], 0
        for k in range(N):
            Hd2 = prmt(X.hB, wv[k], 0x7632)
            Ed2 = prmt(X.EN, wv[k], 0x5432)
            sc = prmt(sl[k >> 2], sg[k >> 2], 0xC480 + (k & 3) * 0x1111)
            M2 = viaddmin_s16x2(Hd2, sc, positive_h2(Hd2))
            h2 = vimax3_s16x2(M2, Ed2, X.F)
            Mi2 = sub_sat_h2(M2, self.oe_i2)
            Md2 = Mi2 if self.sym else sub_sat_h2(M2, self.oe_d2)
            EN2 = viaddmax_s16x2(Ed2, self.ne_d2, Md2)
            X.F = viaddmax_s16x2(X.F, self.ne_i2, Mi2)
            self.S[s + k - 1] = prmt(EN2, X.hA, 0x5410)
            h8 = mul(h2, 8)
            kb = h8 if k == 0 else viaddmax_u16x2(h8, k * 0x10001, kb)
            X.hB, X.hA, X.EN = X.hA, h2, EN2
            hh.append(h2)
        t0, t1 = kb >> 16, kb & 0xffff
        X.k0 = max(X.k0, t0 * 64 - (t0 & 7) * 63 + s)
        X.k1 = max(X.k1, t1 * 64 - (t1 & 7) * 63 + s - 1)
        X.settle(s, hh)


def bound_ok(params, q, t, h0, lane):
    """The kernels' preconditions on a pair's score bound and N bases."""
    bound = h0 + params.scoring.match * min(len(q), len(t))
    has_n = (np.asarray(q) > 3).any() or (np.asarray(t) > 3).any()
    return bound <= 255 if lane is Lane8 else bound <= 2047 and not has_n


def extend(params, q, t, h0, w=None, lane=Lane8, nm=None):
    """One pair through the row-pair pass.  Returns (results dict, cells).

    nm: the lane with N codes (default: whether the pair has an N).
    Preconditions of the kernels' row-pair path: n, m >= 1, and a score bound
    h0 + match * min(n, m) of at most 255 (Lane8) or 2047 (Lane16, no N)."""
    sc = params.scoring
    e_del, e_ins = sc.e_del, sc.e_ins
    oe_del, oe_ins = sc.o_del + e_del, sc.o_ins + e_ins
    n, m = len(q), len(t)
    assert n >= 1 and m >= 1 and bound_ok(params, q, t, h0, lane)
    if nm is None:
        nm = bool((np.asarray(q) > 3).any() or (np.asarray(t) > 3).any())
    wb = oracle.band_width(params, n, params.w if w is None else w)
    V = lane(sc, q, h0, nm)
    KEY = lane.KEY

    def cell(d, e, f, s):
        M = d + s if d > 0 else 0
        return max(M, e, f), max(e - e_del, M - oe_del, 0), max(f - e_ins, M - oe_ins, 0)

    lo, hi = 0, n
    best, bi, bj, gbest, gi, moff = h0, -1, -1, -1, -1, 0
    ncell = 0

    def decide(row, key, lo_r, hi_r, h_end):
        """Row decisions (Section V-D): query-end score, all-zero row, best,
        z-drop.  Returns False to stop."""
        nonlocal best, bi, bj, gbest, gi, moff, ncell
        rm, rj = key // KEY, key % KEY
        if hi_r > lo_r:
            ncell += hi_r - lo_r
        if max(lo_r, hi_r) == n:
            if h_end >= gbest:
                gi = row
            gbest = max(gbest, h_end)
        if rm == 0:
            return False
        if rm > best:
            best, bi, bj = rm, row, rj
            moff = max(moff, abs(rj - row))
        elif params.zdrop > 0:
            di, dj = row - bi, rj - bj
            drop = best - rm - (di - dj) * e_del if di > dj else best - rm - (dj - di) * e_ins
            if drop > params.zdrop:
                return False
        return True

    for i in range(0, m, 2):
        single = i + 1 == m
        V.rows(int(t[i]), 0 if single else int(t[i + 1]))
        lo = max(lo, i - wb)
        hi = min(hi, i + wb + 1, n)
        hl0 = max(0, h0 - oe_del - i * e_del) if lo == 0 else 0
        # Row i alone until its first non-zero slot and row i+1's lower clip.
        f, hprev, hprev2, en_last, key_lo, Lp = 0, hl0, 0, 0, 0, 0
        found, lo1, c0 = False, hi, None
        for s in range(lo, hi):
            d, e = V.get(s)
            h, en, f = cell(d, e, f, V.score0(s))
            key_lo = max(key_lo, h * KEY + s)
            if h > 0:
                Lp = s + 1
            if not found and (hprev | en):
                found, lo1 = True, s
            hprev2, hprev, en_last = hprev, h, en
            if not single and found and s >= max(lo1, i + 1 - wb):
                c0 = s
                break
        if single:
            decide(i, key_lo, lo, hi, hprev if hi > lo else hl0)
            break
        if c0 is None:
            c0 = max(lo1, i + 1 - wb)
        bnd1 = max(0, h0 - oe_del - (i + 1) * e_del) if c0 == 0 else 0
        # Both rows: step s computes (i, s) in the high halves, (i+1, s-1) low.
        X = Row(pack(bnd1, hprev), hprev2 << 16, en_last << 16, f << 16, Lp)
        V.open(X, c0, bnd1, key_lo)
        s = c0 + 1
        while s + 8 <= hi:
            V.steps(s, X, 8)
            s += 8
        rest = max(hi - s, 0)
        for N in (4, 2, 1):
            if rest & N:
                V.steps(s, X, N)
                s += N
        if hi > c0 + 1:
            Hi1, Hi2, Ei1 = X.hA >> 16, X.hB >> 16, X.EN >> 16
            ce, fh, hlh, Lp = hi - 1, X.F & 0xffff, X.hA & 0xffff, X.L
        else:
            Hi1, Hi2, Ei1 = hprev, hprev2, en_last
            ce, fh, hlh = c0, 0, bnd1
        key_lo, key_hi = V.close(X)
        if not decide(i, key_lo, lo, hi, Hi1 if hi > lo else hl0):
            break
        # Row i+1's band is [c0, hi1); its columns from ce on run alone.
        hi1 = min(Lp + 2, n, i + 1 + wb + 1)
        for c in range(ce, hi1):
            if c == hi - 1:
                d, e = Hi2, Ei1
            elif c == hi:
                d, e = Hi1, 0
            else:                   # past row i's end: the slot as it stands
                d, e = V.get(c)
            h, en, fh = cell(d, e, fh, V.score1(c))
            V.put(c, hlh, en)
            key_hi = max(key_hi, h * KEY + c)
            hlh = h
        if hi1 >= ce and hi1 > c0:
            V.put(hi1, hlh, 0)
        if not decide(i + 1, key_hi, c0, hi1, V.h_of(hi1) if hi1 > c0 else bnd1):
            break
        for k in range(hi1 + 1, hi + 1):      # row i's zeros past row i+1's end
            V.put(k, 0, 0)
        k = c0                                 # rule c on row i+1's slots
        while k < hi1 and not V.nonzero(k):
            k += 1
        lo = k
        k = hi1
        while k >= lo and not V.nonzero(k):
            k -= 1
        hi = min(k + 2, n)
    return dict(score=best, qle=bj + 1, tle=bi + 1, gtle=gi + 1, gscore=gbest, max_off=moff), ncell
