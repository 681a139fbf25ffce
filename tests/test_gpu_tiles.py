"""Edges of the warp tiles: curves around the 32-observation chunks, grids around
the tile and anchor-block widths, grids off the line (products with the distance
from an exact phase, blocks on lines of their own, no order, spans too wide for
the products), and the merge of thousands of candidate rows."""
from __future__ import annotations

import numpy as np
import pytest

import lightcurves as L
import oracle
from gpu_util import assert_S_close, bin_mismatches, check_topk, run_batch, run_bins, s_bound, to_dev

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

NS = [1, 3, 4, 5, 31, 32, 33, 63, 64, 65, 97, 0, 129]


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2502_00243_gb300 as G
    c = G.Context(0)
    yield c
    c.close()


def check_batch(ctx, w, M, k, params=None):
    """Dense S (tiles inside anchor blocks) and the top-k of a call with and
    without it, against the oracle."""
    d = to_dev(w)
    _, _, Sd, st = run_batch(ctx, w, M=M, k=0, dense=True, d=d, params=params)
    idx, S, Sk, st2 = run_batch(ctx, w, M=M, k=k, dense=True, d=d, params=params)
    free_idx, free_S, _, st3 = run_batch(ctx, w, M=M, k=k, d=d, params=params)
    assert (st, st2, st3) == (0, 0, 0)
    np.testing.assert_array_equal(Sk, Sd)  # the anchors don't depend on the tiles
    for c in range(w.ncurves):
        t, x, s = w.curve(c)
        S_or = oracle.fpw(t, x, s, w.freqs, M) if t.size else np.zeros(w.nfreq)
        near = oracle.min_edge(t, w.freqs, M) <= 1e-9 if t.size else np.zeros(w.nfreq, bool)
        assert_S_close(Sd[c], S_or, s_bound(x, s), mask=~near, what=f"curve {c} of {t.size}")
        o_idx, o_S = oracle.topk(S_or, k + 4)
        if not near.any():
            for gi, gs in ((idx, S), (free_idx, free_S)):
                check_topk(gi[c], gs[c], o_idx, o_S, abs_tol=1e-7 * s_bound(x, s), o_dense=S_or, what=f"curve {c}")


@pytest.mark.parametrize("M", [1, 7, 16, 20, 33, 50, 64])
@pytest.mark.parametrize("F", [1, 2, 33, 159, 639, 1023, 2050])
def test_chunk_tile_and_block_edges(ctx, M, F):
    w = L.ragged(500 + M, NS, F, M=M, k=3)
    w.freqs = 0.0137 + 0.00311 * np.arange(F)  # f = 0 keeps every observation on an edge
    check_batch(ctx, w, M, 3)


def _grids(F):
    rng = np.random.default_rng(7)
    log = np.geomspace(0.02, 10.0, F)
    two = np.concatenate([0.02 + 1e-4 * np.arange(F // 2), 3.0 + 7e-4 * np.arange(F - F // 2)])
    return {"log": log, "descending": log[::-1].copy(), "two_lines": two, "no_order": rng.permutation(log),
            "wide": np.geomspace(0.02, 500.0, F)}


@pytest.mark.parametrize("accum", [0, 1, 2])
@pytest.mark.parametrize("name", ["log", "descending", "two_lines", "no_order", "wide"])
def test_grids_off_the_line(ctx, name, accum):
    import paper_2502_00243_gb300 as G
    w = L.ragged(520, [700, 33, 64, 5], 10, M=20, k=4)
    w.freqs = _grids(1501)[name]
    check_batch(ctx, w, 20, 4, params=G.fpw_params_default(accum=accum))


@pytest.mark.parametrize("name", ["log", "descending", "two_lines", "no_order", "wide"])
def test_bins_off_the_line(ctx, name):
    w = L.ragged(521, [900, 77], 10, M=20)
    w.t -= 300.0  # negative times too
    w.freqs = _grids(2003)[name]
    g, _, st = run_bins(ctx, w, 0, w.nfreq)
    assert st == 0
    pairs, _, far, _ = bin_mismatches(g, w, 0, w.nfreq, 20, oracle.bins)
    assert pairs == w.nfreq * w.nobs and far == 0


@pytest.mark.parametrize("k", [1, 5, 64])
def test_peaks_of_a_curve_in_thousands_of_rows(ctx, k):
    """The merged list is exactly the list of the dense values' peaks."""
    import paper_2502_00243_gb300 as G
    w = L.ragged(530, [40], 600_000, M=8, k=k)
    d = to_dev(w)
    for params in (None, G.fpw_params_default(items_per_slot=64, threads=32, freqs_per_thread=1)):
        idx, S, Sd, st = run_batch(ctx, w, d=d, dense=True, params=params)
        assert st == 0
        o_idx, o_S = oracle.topk(Sd[0], k)
        np.testing.assert_array_equal(idx[0], o_idx)
        np.testing.assert_array_equal(S[0], o_S.astype(np.float32))
