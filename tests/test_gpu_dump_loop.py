"""The dumped bins are those of the sums: with binary64 bins, whose additions and
terms round once each in the order of the observations and bins, the periodogram
of the call without a dump follows from the dumped bins bit for bit, in every way
of forming the bins (steps from anchors, products off the line, exact pairs, FP32
phases)."""
from __future__ import annotations

import numpy as np
import pytest

import lightcurves as L
import oracle
from gpu_util import run_batch, run_bins, to_dev

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

GRIDS = {"line": lambda F: 0.25 + 5e-4 * np.arange(F), "log": lambda F: np.geomspace(2.0, 4.0, F),
         "wide": lambda F: np.geomspace(0.02, 4000.0, F), "negative": lambda F: -0.3 + 5e-4 * np.arange(F)}


@pytest.mark.parametrize("phase", [0, 2])
@pytest.mark.parametrize("M", [7, 20])
@pytest.mark.parametrize("grid", sorted(GRIDS))
def test_values_follow_from_the_dumped_bins(grid, M, phase):
    import paper_2502_00243_gb300 as G
    ctx = G.Context(0)
    w = L.ragged(3, [65, 130, 1, 31], 2, M=M, k=4)
    w.t[:65] = np.round(w.t[:65] * 48) / 48
    w.freqs = GRIDS[grid](1111)
    p, d = G.fpw_params_default(accum=1, phase_mode=phase, K=100), to_dev(w)
    bins, _, st = run_bins(ctx, w, 0, w.nfreq, params=p, d=d)
    assert st == 0 and (bins >= 0).all() and (bins < M).all()
    _, _, Sd, _ = run_batch(ctx, w, k=0, dense=True, params=p, d=d)
    idx, S, _, _ = run_batch(ctx, w, params=p, d=d)
    for c in range(w.ncurves):
        o0, o1 = int(w.offsets[c]), int(w.offsets[c + 1])
        wt = 1.0 / (w.sigma[o0:o1] * w.sigma[o0:o1])
        a, rows = w.x[o0:o1] * wt, np.arange(w.nfreq)
        A, B, want = np.zeros((w.nfreq, M)), np.zeros((w.nfreq, M)), np.zeros(w.nfreq)
        for i in range(o1 - o0):
            A[rows, bins[:, o0 + i]] += a[i]
            B[rows, bins[:, o0 + i]] += wt[i]
        for m in range(M):
            q = B[:, m] > 0
            want[q] += A[q, m] * A[q, m] / B[q, m]
        np.testing.assert_array_equal(Sd[c], want)
        o_idx, o_S = oracle.topk(want, 4)
        np.testing.assert_array_equal(idx[c], o_idx)
        np.testing.assert_array_equal(S[c], o_S.astype(np.float32))
    ctx.close()
