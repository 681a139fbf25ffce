"""The phases behind a list of peaks are those of the dense periodogram: a call's
lists are exactly the peaks of its dense values, with and without dense output, in
a batch and alone, with scratch of its own or none to allocate. Visits thirty
minutes apart at round frequencies put phases on bin edges, where an anchor or a
step that differs by 1e-16 cycles moves observations to other bins.

And the bins are those of exact arithmetic on the rounded anchors and steps: the
anchor's phase and the step are the exact products rounded up at 2^-64, a bin is
floor(M floor(2^32 phase) / 2^32) of the anchor's phase plus whole steps."""
from __future__ import annotations

from fractions import Fraction

import numpy as np
import pytest

import lightcurves as L
import oracle
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


def on_edges(seed, ns, F, df, M, k):
    """Curves whose visits lie on multiples of 30 minutes, or 30 minutes after visits at any time."""
    w = L.ragged(seed, ns, F, M=M, k=k)
    rng = np.random.default_rng(seed)
    for c in range(w.ncurves):
        o0, o1 = int(w.offsets[c]), int(w.offsets[c + 1])
        n = o1 - o0
        if c % 2:
            w.t[o0:o1] = np.sort(rng.integers(0, 48 * 700, n)) / 48.0
        else:
            first = rng.integers(0, 700, n) + 0.1 + 0.3 * rng.random(n)
            t = np.sort(np.concatenate([first, first + 1 / 48])[:n])
            w.t[o0:o1] = t - (t[0] if n else 0.0)
    w.freqs = df * np.arange(F)
    return w


@pytest.mark.parametrize("df", [5e-4, 2.5e-4, 1 / 4096])
@pytest.mark.parametrize("M", [8, 10, 16, 20, 30, 50, 60, 90])
def test_lists_are_the_peaks_of_the_dense_values(ctx, M, df):
    import paper_2502_00243_gb300 as G
    w = on_edges(40 + M, [60, 61, 700, 333, 90, 5, 1, 0], 20001, df, M, 6)
    d = to_dev(w)
    _, _, Sd, st = run_batch(ctx, w, k=0, dense=True, d=d)
    assert st == 0
    o = [oracle.topk(Sd[c], 6) for c in range(w.ncurves)]
    want_i, want_S = np.stack([q[0] for q in o]), np.stack([q[1] for q in o]).astype(np.float32)
    for params, dense in ((None, False), (None, True), (G.fpw_params_default(items_per_slot=64), False)):
        idx, S, _, st = run_batch(ctx, w, d=d, dense=dense, params=params)
        assert st == 0
        np.testing.assert_array_equal(idx, want_i)
        np.testing.assert_array_equal(S, want_S)
    raw = [oracle.topk(Sd[c], 6, raw=True) for c in range(w.ncurves)]
    idx, S, _, _ = run_batch(ctx, w, d=d, params=G.fpw_params_default(peak_mode=1))
    np.testing.assert_array_equal(idx, np.stack([q[0] for q in raw]))
    np.testing.assert_array_equal(S, np.stack([q[1] for q in raw]).astype(np.float32))


@pytest.mark.parametrize("accum", [0, 1, 2])
def test_lists_do_not_depend_on_the_call_around_a_curve(ctx, accum):
    """A curve alone, next to one of long times, and without allocation (at the same anchors)."""
    import paper_2502_00243_gb300 as G
    w = on_edges(7, [400, 401, 64], 20001, 5e-4, 20, 5)
    p = G.fpw_params_default(accum=accum, threads=128, freqs_per_thread=2)
    idx, S, _, _ = run_batch(ctx, w, params=p)
    for c in range(w.ncurves):
        one = L.ragged(1, [1], 2, M=20, k=5)
        t, x, s = w.curve(c)
        one.t, one.x, one.sigma, one.freqs = t, x, s, w.freqs
        one.offsets = np.array([0, t.size], np.int64)
        i1, S1, _, _ = run_batch(ctx, one, params=p)
        np.testing.assert_array_equal(i1[0], idx[c])
        np.testing.assert_array_equal(S1[0], S[c])
    far = L.ragged(2, [1], 2, M=20, k=5)
    far.t, far.x, far.sigma = (np.concatenate([a, b]) for a, b in
                               ((w.t, 1e9 + 1e6 * np.arange(40.0)), (w.x, np.ones(40)), (w.sigma, np.ones(40))))
    far.freqs, far.offsets = w.freqs, np.concatenate([w.offsets, w.offsets[-1:] + 40])
    i2, S2, _, _ = run_batch(ctx, far, params=p)
    np.testing.assert_array_equal(i2[:3], idx)
    np.testing.assert_array_equal(S2[:3], S)
    d = to_dev(w)
    i3 = torch.empty(15, dtype=torch.int32, device="cuda")
    S3 = torch.empty(15, dtype=torch.float32, device="cuda")
    G.fpw_periodogram_batch_noalloc(None, p, d["offsets"], w.offsets, d["t"], d["x"], d["sigma"], d["freqs"], 20, 5, i3, S3)
    np.testing.assert_array_equal(i3.cpu().numpy().reshape(3, 5), idx)
    np.testing.assert_array_equal(S3.cpu().numpy().reshape(3, 5), S)


@pytest.mark.parametrize("Mx,groups", [(60, [3, 6, 15]), (40, [2, 4, 10]), (20, [1, 2, 4]), (36, [2, 3, 6])])
def test_several_M_lists(ctx, Mx, groups):
    import paper_2502_00243_gb300 as G
    w = on_edges(90 + Mx, [60, 501, 700], 12001, 5e-4, Mx, 4)
    d, C, ng, F, k = to_dev(w), 3, len(groups), 12001, 4

    def run(dense):
        idx = torch.empty(C * ng * k, dtype=torch.int32, device="cuda")
        off, S = torch.empty_like(idx), torch.empty(C * ng * k, dtype=torch.float32, device="cuda")
        Sd = torch.empty(C * ng * F, dtype=torch.float64, device="cuda") if dense else None
        G.fpw_periodogram_batch_multi(ctx, None, None, d["offsets"], w.offsets, d["t"], d["x"], d["sigma"], d["freqs"],
                                      Mx, groups, k, idx, off, S, Sd)
        assert ctx.status() == 0
        return idx.cpu().numpy().reshape(-1, k), off.cpu().numpy(), S.cpu().numpy().reshape(-1, k), Sd

    i0, o0, S0, _ = run(False)
    i1, o1, S1, Sd = run(True)
    np.testing.assert_array_equal(i0, i1)
    np.testing.assert_array_equal(o0, o1)
    np.testing.assert_array_equal(S0, S1)
    for row, Sr in enumerate(Sd.cpu().numpy().reshape(-1, F)):
        o_idx, o_S = oracle.topk(Sr, k)
        np.testing.assert_array_equal(i0[row], o_idx)
        np.testing.assert_array_equal(S0[row], o_S.astype(np.float32))


def _up(v):
    """ceil(frac(v) 2^64) mod 2^64."""
    n = v.numerator << 64
    return -((-n) // v.denominator) & (2 ** 64 - 1)


@pytest.mark.parametrize("name", ["visits", "mjd", "negative", "seconds", "small", "mixed", "below_zero"])
def test_bins_step_from_exact_anchors(ctx, name):
    import paper_2502_00243_gb300 as G
    rng = np.random.default_rng(3)
    n, F, M, T, R = 50, 1100, 20, 64, 4
    t = np.sort(rng.integers(0, 48 * 900, n)) / 48.0
    t[:20] += rng.random(20)
    f = 5e-4 * np.arange(F) + 2.99
    if name == "mjd":
        t = t + 58000.0
    elif name == "negative":
        t = t - 450.0
    elif name == "seconds":
        t, f = t * 86400.0, f / 86400.0
    elif name == "small":
        t, f = t * 2.0 ** -40, f * 2.0 ** 40
    elif name == "mixed":  # times that the call's fixed-point format holds and others
        t = np.concatenate([t[:25], t[25:] * 2.0 ** -60])
    elif name == "below_zero":
        f = f - 3.1
    w = L.ragged(1, [n], 2, M=M, k=1)
    w.t, w.freqs = t, f
    g, _, st = run_bins(ctx, w, 0, F, params=G.fpw_params_default(threads=T, freqs_per_thread=R))
    assert st == 0
    A, df = T * R - 2, float((f[-1] - f[0]) / (F - 1))
    want = np.empty((F, n), np.int64)
    for i, ti in enumerate(map(Fraction, t.tolist())):
        D = _up(ti * Fraction(df))
        for q in range(-(-F // A)):
            a = max(q * A - 1, 0)
            P = _up(ti * Fraction(float(f[a])))
            for k in range(q * A, min((q + 1) * A, F)):
                want[k, i] = M * ((P + (k - a) * D & 2 ** 64 - 1) >> 32) >> 32
    np.testing.assert_array_equal(g, want)
