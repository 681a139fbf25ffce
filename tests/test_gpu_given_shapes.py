"""Shapes that a caller gives: those with the same product of threads and
frequencies per thread have the same phase anchors, hence the same S and peaks bit
for bit, whatever blocks their warps are launched in."""
from __future__ import annotations

import numpy as np
import pytest

import lightcurves as L
from gpu_util import run_batch, to_dev

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("accum", [0, 2])
@pytest.mark.parametrize("M", [7, 20, 50])
@pytest.mark.parametrize("T", [32, 96, 160, 224, 256, 288, 480, 512])
def test_same_anchors_same_results(T, M, accum):
    import paper_2502_00243_gb300 as G

    w = L.ragged(T + M, [300, 0, 33, 1, 90], 3001, M=M, k=4)
    w.t[:300] = np.round(w.t[:300] * 48) / 48
    d, ctx, ran = to_dev(w), G.Context(0), []
    for R in (1, 2, 4, 8):
        if T % (32 * R) == 0:
            try:
                ran.append(run_batch(ctx, w, params=G.fpw_params_default(threads=T // R, freqs_per_thread=R, accum=accum),
                                     dense=True, d=d))
            except G.FPWError:
                assert T * M * (8 if accum == 0 else 16) > 100_000  # only where a block's bins are large
    for r in ran:
        assert r[3] == 0
        for a, b in zip(r[:3], ran[0][:3]):
            np.testing.assert_array_equal(a, b)
    assert ran or T * M * (8 if accum == 0 else 16) > 200_000
