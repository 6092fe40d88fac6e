"""The per-thread kernels on small batches (needs a GPU).

Batches of up to 12,288 pairs run their queries of up to 256 bases one per warp
(k_short), so the row-pair, N-base and plan cases, which are small, would no
longer reach the per-thread kernels they were written for.  Kernel timing asks
for the plan's own kernels; these tests run the same cases with it.  The last
one runs k_short against them at its own edges: every number of columns per
lane, and query lengths at the lanes' ends.
"""
import numpy as np
import pytest

import oracle
import test_gpu_nbase as nbase
import test_gpu_plan as plan
import test_gpu_rowpair as rowpair
from paper_1907_12931_gb300 import workload as W
from test_gpu_parity import NTH, assert_same, run

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def bsw():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1907_12931_gb300 import bsw as _b
    _b.lib()
    return _b


@pytest.fixture
def timed(bsw, monkeypatch):
    """The three modules' runs with kernel timing, hence on the plan's kernels."""
    def flagged(flags, device):
        return flags | bsw.BSW_TIME_KERNELS | (bsw.BSW_NO_GRAPH if device else 0)

    def timed_run(b, wl, flags=0, device=False, **kw):
        return run(b, wl, flags=flagged(flags, device), device=device, **kw)

    run_plan = plan.run_plan

    def timed_plan(b, wl, p, flags=0, device=False, **kw):
        return run_plan(b, wl, p, flags=flagged(flags, device), device=device, **kw)

    monkeypatch.setattr(rowpair, "run", timed_run)
    monkeypatch.setattr(nbase, "run", timed_run)
    monkeypatch.setattr(plan, "run_plan", timed_plan)
    return bsw


@pytest.mark.parametrize("k", range(len(rowpair.SCORINGS)))
def test_random_pairs(timed, k):
    rowpair.test_random_pairs(timed, k)


@pytest.mark.parametrize("w", [1, 2, 3, 5, 8])
def test_stale_slot_reads(timed, w):
    rowpair.test_stale_slot_reads(timed, w)


def test_row_counts(timed):
    rowpair.test_row_counts(timed)


def test_score_bound_edges(timed):
    rowpair.test_score_bound_edges(timed)


@pytest.mark.parametrize("p", plan.PLANS, ids=[str(sorted(p.items())) for p in plan.PLANS])
def test_plan_parity_adversarial(timed, p):
    plan.test_plan_parity_adversarial(timed, p)


def test_hand_cases_with_n(timed):
    nbase.test_hand_cases(timed, 0)


@pytest.mark.parametrize("zdrop", [100, 0, 7])
def test_adversarial_with_n(timed, zdrop):
    nbase.test_adversarial_with_n(timed, zdrop, 0)


@pytest.mark.parametrize("sc,w,zd", [((1, 4, 6, 1, 6, 1), 100, 100), ((2, 8, 12, 2, 12, 2), 100, 200),
                                     ((1, 4, 6, 1, 6, 1), 3, 0), ((3, 5, 4, 2, 7, 1), 9, 30), ((127, 128, 0, 1, 0, 1), 20, 0)])
@pytest.mark.parametrize("n_rate", [0.0, 0.04])
def test_row_in_registers(bsw, sc, w, zd, n_rate):
    rng = np.random.default_rng(sc[0] * 1000 + w)
    qs, ts, hs = [], [], []
    for n in (1, 2, 3, 4, 5, 31, 32, 33, 63, 64, 65, 127, 128, 129, 131, 155, 159, 160, 161, 186, 191, 192, 193, 249, 255, 256):
        for m in (1, 2, 3, n, n + 3, n + 100, 2 * n + 1):
            ref = rng.integers(0, 4, n + m + 8)
            q = np.where(rng.random(n) < rng.choice([0.0, 0.05, 0.4]), rng.integers(0, 4, n), ref[:n])
            t = ref[int(rng.integers(0, 5)):][:m] if rng.random() < 0.8 else rng.integers(0, 4, m)
            q[rng.random(n) < n_rate] = 4
            t[rng.random(m) < n_rate] = 4
            for h0 in (0, 9, 60, 200, 900):
                qs.append(q.astype(np.uint8)); ts.append(t.astype(np.uint8)); hs.append(h0)
    wl = W.from_lists(qs, ts, hs, W.Params(W.Scoring(*sc), w=w, zdrop=zd, end_bonus=5), align=4)
    assert wl.n_pairs < 12288
    ref, cells, _ = oracle.extend_batch(wl, nthreads=NTH)
    for flags in (0, bsw.BSW_TIME_KERNELS | bsw.BSW_NO_GRAPH):
        got, gc = run(bsw, wl, flags=flags, device=True)
        assert_same(got, ref, "%s w=%d flags %d" % (sc, w, flags))
        assert gc == int(cells.sum())
