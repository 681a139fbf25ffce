"""Lists of peaks on both sides of where a curve's candidates are merged by a block
or by a warp: numbers of curves around whole rounds of blocks, few and many peaks,
one long curve among short ones. The lists are the peaks of the dense values."""
from __future__ import annotations

import numpy as np
import pytest

import lightcurves as L
import oracle
from gpu_util import run_batch, to_dev

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k", [1, 5, 64])
@pytest.mark.parametrize("C,long", [(1, 900), (2, 30), (20, 30), (152, 30), (153, 30), (304, 5), (305, 2000), (900, 2000)])
def test_lists_are_the_peaks_of_the_dense_values(C, long, k):
    import paper_2502_00243_gb300 as G

    w = L.ragged(C + k, [long] + [3 + c % 28 for c in range(1, C)], 2003, M=10, k=k)
    d, ctx = to_dev(w), G.Context(0)
    _, _, Sd, st = run_batch(ctx, w, k=0, dense=True, d=d)
    idx, S, _, st2 = run_batch(ctx, w, d=d)
    assert st == 0 and st2 == 0
    want = [oracle.topk(r, k) for r in Sd]
    np.testing.assert_array_equal(idx, np.stack([q[0] for q in want]))
    np.testing.assert_array_equal(S, np.stack([q[1] for q in want]).astype(np.float32))
