"""items_per_slot bounds the work items from below, up to the largest int: the
work list is as long as there are tiles, and the lists of peaks are those of the
tuned schedule."""
from __future__ import annotations

import numpy as np
import pytest

import lightcurves as L
from gpu_util import run_batch

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("items", [1, 1000, 2 ** 31 - 1])
def test_any_number_of_items_per_slot(items):
    import paper_2502_00243_gb300 as G

    ctx = G.Context(0)
    w = L.ragged(8, [300, 0, 41, 1], 5003, M=20, k=3)
    want = run_batch(ctx, w)
    got = run_batch(ctx, w, params=G.fpw_params_default(items_per_slot=items))
    assert want[3] == got[3] == 0
    np.testing.assert_array_equal(got[0], want[0])
    np.testing.assert_array_equal(got[1], want[1])
    ctx.set_shape(20, 20, 0, 10 ** 6, 128, 4, 0, items)
    assert run_batch(ctx, w)[3] == 0
