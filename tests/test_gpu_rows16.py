"""The 16-bit per-thread kernel's row pairs against the oracle (needs a GPU).

Pairs of the 16-bit classes up to a score bound of 2047 run two rows per
packed instruction, the others one row at a time.  The cases sit at that line
(h0 + match * min(n, m) at 2046 to 2049), at the code words' and blocks' edges
(query lengths around multiples of 8, and each class's bound), and at row
counts of one to nine.  Every comparison is bit-exact on all six result fields
and the cell count.
"""
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
