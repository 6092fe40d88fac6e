"""The SMEM search's two kernels at their edges (needs a GPU).

k_smem_scan takes groups of 32 reads and notes the searches' starts,
k_smem_store works them off, in as many rounds as the budget's room for starts
takes.  Cases: read counts around a group, empty and one-base reads, reads
unrelated to the text (a start every dozen bases), budgets that hold the starts
of a few reads at a time, one long read among short ones, and starts given up
for other calls.
"""
import numpy as np
import pytest

from oracle import smem as oracle_smem
from paper_1907_12931_gb300 import workload as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def bsw():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1907_12931_gb300 import bsw as _b
    _b.lib()
    return _b


def make_reads(rng, ref, n, lmax):
    out = []
    for k in range(n):
        ln = int(rng.choice([0, 1, 2, 40, lmax]))
        p = int(rng.integers(0, len(ref) - lmax))
        x = ref[p:p + ln].copy() if k % 3 else rng.integers(0, 4, ln).astype(np.uint8)
        x[rng.random(ln) < 0.03] = 2
        out.append(np.ascontiguousarray(3 - x[::-1]) if k & 1 else x)
    return out


def search(bsw, ctx, reads, min_len):
    ln = np.array([len(x) for x in reads], np.int32)
    off, total = W.layout(ln, 4)
    codes = np.zeros(total, np.uint8)
    for o, x in zip(off, reads):
        codes[o:o + len(x)] = x
    rec, first = ctx.smem(bsw.bsw_pack_2bit(codes), off, ln, min_len=min_len)
    return [[tuple(int(rec[f][k]) for f in ("qbeg", "len", "k", "s")) for k in range(first[r], first[r + 1])]
            for r in range(len(reads))]


def expected(ref, reads, min_len):
    return [[tuple(int(v) for v in rec) for rec in r] for r in oracle_smem.smems(ref, reads, min_len)]


@pytest.mark.parametrize("n", [1, 31, 32, 33, 64, 97])
def test_group_edges(bsw, n):
    rng = np.random.default_rng(n)
    ref = rng.integers(0, 4, 1500).astype(np.uint8)
    reads = make_reads(rng, ref, n, 130)
    with bsw.Context(W.Params(), 1 << 30) as ctx:
        ctx.fm_build(ref)
        for min_len in (1, 7):
            assert search(bsw, ctx, reads, min_len) == expected(ref, reads, min_len)


def rounds_of(bsw, call):
    """Rounds of a search: as many of its launches as an injected failure can skip."""
    for k in range(1, 1000):
        assert bsw.bsw_fault_inject("launch:%d" % k) == bsw.BSW_OK
        try:
            call()
        except bsw.BswError as e:
            assert e.code == bsw.BSW_ECUDA
            continue
        finally:
            bsw.bsw_fault_inject(None)
        return k


def test_rounds_under_a_tight_budget(bsw):
    """Budgets down to the least that holds the reads and their records: the
    search then runs in rounds, with reads on both sides of a round's end in one
    group of 32.  No read needs lists or has more records than are kept."""
    rng = np.random.default_rng(8)
    ref = rng.integers(0, 4, 2000).astype(np.uint8)
    reads = make_reads(rng, ref, 301, 600)
    want = expected(ref, reads, 50)
    assert 0 < max(len(r) for r in want) <= 8
    seen = set()
    for budget in list(range(60_000, 200_000, 3_000)) + [1 << 22]:
        with bsw.Context(W.Params(), budget) as ctx:
            try:
                ctx.fm_build(ref)
                got = search(bsw, ctx, reads, 50)
            except bsw.BswError as e:
                assert e.code == bsw.BSW_EBUDGET and not seen
                continue
            assert got == want
            seen.add(rounds_of(bsw, lambda: search(bsw, ctx, reads, 50)))
            assert search(bsw, ctx, reads, 50) == want
    assert 1 in seen and 2 in seen and max(seen) >= 5, seen


def long_among_short():
    """20 000 reads of 60 bases, 40 of them with some ten records, and one of 32 768."""
    rng = np.random.default_rng(5)
    ref = rng.integers(0, 4, 50_000).astype(np.uint8)
    reads = [ref[p:p + 60].copy() for p in rng.integers(0, 49_000, 20_000)]
    for x in reads[:40]:
        x[::6] = (x[::6] + 1) % 4
    one = rng.integers(0, 4, 32768).astype(np.uint8)
    one[:30000] = ref[:30000]
    return ref, reads[:7000] + [one] + reads[7000:]


def test_one_long_read_among_short_ones(bsw):
    """The long read takes room for its own starts, not for every group's, and
    the lists of the reads with many records find their room: 40 MB hold the
    call, as they hold the reads, their records and 41 lists."""
    ref, reads = long_among_short()
    with bsw.Context(W.Params(), 1 << 30) as ctx:
        ctx.fm_build(ref)
        want = search(bsw, ctx, reads, 4)
    few = [k for k in range(len(reads)) if k % 500 == 0 and len(reads[k]) < 100] + [3, 39]
    assert [want[k] for k in few] == expected(ref, [reads[k] for k in few], 4)
    assert sum(len(r) > 8 for r in want) >= 40
    with bsw.Context(W.Params(), 40 << 20) as ctx:
        ctx.fm_build(ref)
        for _ in range(2):                                         # the second with the first's lists still held
            assert search(bsw, ctx, reads, 4) == want


def test_starts_are_given_up(bsw):
    """Where an allocation is refused, the starts an earlier search left make
    room for it; a search does with half the starts where theirs is refused."""
    rng = np.random.default_rng(10)
    ref = rng.integers(0, 4, 2000).astype(np.uint8)
    reads = make_reads(rng, ref, 200, 130)
    want = expected(ref, reads, 12)
    sa = np.arange(3_000_000, dtype=np.int32)
    with bsw.Context(W.Params(), 1 << 30) as ctx:
        ctx.fm_build(ref)
        assert search(bsw, ctx, reads, 12) == want
        try:
            bsw.bsw_fault_inject("alloc")
            ctx.sal_set_index(sa[:1_000_000])                      # refused once: the starts go, and it passes
            bsw.bsw_fault_inject("alloc")
            with pytest.raises(bsw.BswError) as e:                 # nothing left to give up
                ctx.sal_set_index(sa)
            assert e.value.code == bsw.BSW_ENOMEM
        finally:
            bsw.bsw_fault_inject(None)
        assert search(bsw, ctx, reads, 12) == want
    with bsw.Context(W.Params(), 1 << 30) as ctx:
        ctx.fm_build(ref)
        try:
            bsw.bsw_fault_inject("alloc:1")                        # the staging buffer passes, the starts do not
            assert search(bsw, ctx, reads, 12) == want
        finally:
            bsw.bsw_fault_inject(None)
        assert rounds_of(bsw, lambda: search(bsw, ctx, reads, 12)) == 1


@pytest.mark.parametrize("lmax,budget", [(160, 1 << 30), (161, 1 << 30), (300, 1 << 30), (300, 3 << 20)])
def test_reads_with_many_records(bsw, lmax, budget):
    """Counts on both sides of the records a read keeps (8, or 16 past 160
    bases and with room in the budget): the others are searched again."""
    rng = np.random.default_rng(lmax)
    ref = rng.integers(0, 4, 3000).astype(np.uint8)
    reads = []
    for k in range(200):
        p = int(rng.integers(0, len(ref) - lmax))
        x = ref[p:p + lmax].copy()
        at = rng.choice(lmax, int(rng.integers(0, 24)), replace=False)
        x[at] = (x[at] + 1) % 4
        reads.append(np.ascontiguousarray(3 - x[::-1]) if k & 1 else x)
    want = expected(ref, reads, 8)
    counts = [len(r) for r in want]
    assert min(counts) <= 8 < max(counts) and max(counts) > 16
    with bsw.Context(W.Params(), budget) as ctx:
        ctx.fm_build(ref)
        assert search(bsw, ctx, reads, 8) == want


def test_refused_lists_leave_nothing_in_flight(bsw):
    """A call that cannot hold the lists of the reads with many records returns
    with first[] complete, also when it is pinned and the device writes it."""
    import torch
    rng = np.random.default_rng(9)
    ref = rng.integers(0, 4, 3000).astype(np.uint8)
    n = 2_000_000                                                  # 16 MB of first[]
    reads = []
    for _ in range(300):
        p = int(rng.integers(0, 2400))
        x = ref[p:p + 600].copy()
        x[::12] = (x[::12] + 1) % 4                                # some 50 records
        reads.append(x)
    reads.append(rng.integers(0, 4, 32768).astype(np.uint8))       # room for 32769 matches a list
    ln = np.zeros(n, np.int32)
    ln[:len(reads)] = [len(x) for x in reads]
    off, total = W.layout(ln, 4)
    codes = np.zeros(total, np.uint8)
    for o, x in zip(off, reads):
        codes[o:o + len(x)] = x
    packed = bsw.bsw_pack_2bit(codes)
    out, found = np.zeros(100_000, bsw.SMEM_DTYPE), np.zeros(1, np.int64)
    first = torch.full((n + 1,), -1, dtype=torch.int64).pin_memory()
    f = first.numpy()

    def call(ctx):
        return bsw.lib().bsw_smem(ctx.handle, n, packed.ctypes.data, off.ctypes.data, ln.ctypes.data, 10,
                                  out.ctypes.data, out.shape[0], found.ctypes.data, f.ctypes.data)

    with bsw.Context(W.Params(), 4 << 30) as ctx:
        ctx.fm_build(ref)
        assert call(ctx) == bsw.BSW_OK
    want = f.copy()
    with bsw.Context(W.Params(), 400 << 20) as ctx:
        ctx.fm_build(ref)
        for _ in range(5):
            first.fill_(-1)
            assert call(ctx) == bsw.BSW_EBUDGET                    # 300 lists of 32769 entries: 118 MB
            last = int(f[n])
            assert last == found[0] == want[n]
            np.testing.assert_array_equal(f, want)
