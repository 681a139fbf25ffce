"""Grids off the line: the bins are those of the exact phases, floor(M floor(2^32 p)
/ 2^32) with p = ceil(2^64 frac(t f)) / 2^64, for every pair and every way of
cutting the grid into tiles; visits thirty minutes apart at round frequencies put
exact phases just below bin edges, where a phase rounded up by 2^-36 goes wrong."""
from __future__ import annotations

from fractions import Fraction

import numpy as np
import pytest

import lightcurves as L
from gpu_util import run_batch, run_bins, to_dev

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2502_00243_gb300 as G
    c = G.Context(0)
    yield c
    c.close()


def grids(F):
    rng = np.random.default_rng(11)
    f = (1 + np.arange(F)) / 1000.0
    f[1::7] += 2.0 ** -20  # off the line within every block, by little
    return {"round": f, "no_order": rng.permutation(f), "log": np.geomspace(0.02, 10.0, F),
            "negative": f - 0.3, "wide": np.geomspace(0.02, 4000.0, F)}


def times(n, shift=0.0):
    rng = np.random.default_rng(12)
    t = np.sort(rng.integers(0, 48 * 700, n)) / 48.0
    t[0] = 0.0
    t[n // 2:] += rng.random(n - n // 2)
    return t + shift


@pytest.mark.parametrize("M", [8, 20, 33])
@pytest.mark.parametrize("name", ["round", "no_order", "log", "negative", "wide"])
def test_bins_are_those_of_the_exact_phases(ctx, name, M):
    n, F = 70, 700
    w = L.ragged(1, [n], 2, M=M, k=1)
    w.t, w.freqs = times(n, -100.0 if M == 33 else 0.0), grids(F)[name]
    g, _, st = run_bins(ctx, w, 0, F)
    assert st == 0
    mask, want = 2 ** 64 - 1, np.empty((F, n), np.int64)
    fs = [Fraction(v) for v in w.freqs.tolist()]
    for i, ti in enumerate(map(Fraction, w.t.tolist())):
        for k, fk in enumerate(fs):
            v = ti * fk
            want[k, i] = M * ((-((-v.numerator << 64) // v.denominator) & mask) >> 32) >> 32
    np.testing.assert_array_equal(g, want)


@pytest.mark.parametrize("accum", [0, 1, 2])
@pytest.mark.parametrize("name", ["round", "no_order", "log"])
def test_values_do_not_depend_on_the_tiles(ctx, name, accum):
    import paper_2502_00243_gb300 as G
    M, F = 16, 3000
    w = L.ragged(2, [300, 301, 40], 2, M=M, k=7)
    for c in range(3):
        o0, o1 = int(w.offsets[c]), int(w.offsets[c + 1])
        w.t[o0:o1] = times(o1 - o0)
    w.freqs = grids(F)[name]
    d = to_dev(w)
    got = [run_batch(ctx, w, d=d, dense=dense, params=G.fpw_params_default(accum=accum, threads=T, freqs_per_thread=R))
           for T, R in ((256, 1), (128, 2), (64, 4), (32, 8)) for dense in (True, False)]
    for idx, S, Sd, st in got:
        assert st == 0
        np.testing.assert_array_equal(idx, got[0][0])
        np.testing.assert_array_equal(S, got[0][1])
        if Sd is not None:
            np.testing.assert_array_equal(Sd, got[0][2])
    for c in range(3):
        one = L.ragged(1, [1], 2, M=M, k=7)
        one.t, one.x, one.sigma = w.curve(c)
        one.freqs, one.offsets = w.freqs, np.array([0, one.t.size], np.int64)
        idx, S, _, _ = run_batch(ctx, one, params=G.fpw_params_default(accum=accum))
        np.testing.assert_array_equal(idx[0], got[0][0][c])
        np.testing.assert_array_equal(S[0], got[0][1][c])
