"""The long-query kernel's rows in registers against the oracle (needs a GPU).

A pair of the two-columns warp kernel keeps its row in registers when its band
is at most 503 columns to a side and Eq. 3's first row is zero past the band;
the others keep it in the shared-memory ring.  Both must give the oracle's
results and cells, on either side of those lines; with bands that outgrow the
512-column window, shrink back into it and jump past several of its half lanes;
and with rows that end on every column of a half lane.
"""
import numpy as np
import pytest

import oracle
from paper_1907_12931_gb300 import workload as W
from test_gpu_parity import NTH
from test_gpu_warp2 import X2, bsw, check, mutated  # noqa: F401 (bsw is a fixture)

pytestmark = pytest.mark.gpu


def pairs(rng, lengths, h0s, err):
    qs, ts, hs = [], [], []
    for n in lengths:
        ref = rng.integers(0, 4, n + 700)
        gap = int(rng.integers(1, 300))
        cut = int(rng.integers(0, n))
        t = np.concatenate([ref[:cut], ref[cut + gap:], ref[:0]]) if rng.random() < 0.5 else \
            np.concatenate([ref[:cut], rng.integers(0, 4, gap), ref[cut:]])
        qs.append(np.asarray(mutated(rng, ref, n, err))[:n])
        ts.append(t[: max(1, n + int(rng.integers(-min(n - 1, 200), 200)))])
        hs.append(int(rng.choice(h0s)))
    return qs, ts, hs


@pytest.mark.parametrize("w", [0, 1, 7, 8, 100, 230, 244, 500, 502, 503, 504])
@pytest.mark.parametrize("scoring,zdrop", [((1, 4, 6, 1, 6, 1), 100), ((1, 4, 6, 1, 6, 1), 0), ((2, 5, 4, 2, 7, 1), 300),
                                           ((3, 4, 6, 2, 5, 3), 90)])
def test_bands(bsw, w, scoring, zdrop):  # noqa: F811
    rng = np.random.default_rng(700 + w)
    lengths = list(rng.integers(65, 400, 20)) + list(rng.integers(400, 1500, 24)) + [512, 1023, 1024, 2600]
    qs, ts, hs = pairs(rng, lengths, [0, 1, 30, 120, w + 6, w + 8, 700, 2500], 0.05)
    wl = W.from_lists(qs, ts, hs, W.Params(W.Scoring(*scoring), w=w, zdrop=zdrop, end_bonus=5))
    check(bsw, wl, X2, f"w {w}")


def test_band_per_pair(bsw):  # noqa: F811
    rng = np.random.default_rng(811)
    lengths = [int(x) for x in np.linspace(65, 1200, 60)]
    qs, ts, hs = pairs(rng, lengths, [0, 40, 600, 1500], 0.1)
    wl = W.from_lists(qs, ts, hs, W.Params(w=500, zdrop=200))
    wo = rng.choice([0, 5, 200, 500, 503, 504, 700], len(lengths)).astype(np.int32)
    check(bsw, wl, X2, "band per pair", w_override=wo)
