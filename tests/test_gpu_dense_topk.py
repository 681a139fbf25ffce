"""The peaks of the dense FP32 periodogram (curves at common times, drift) against
a sort of the dense values that the same call returns: k from 1 to 64, frequency
counts around a warp's step and a block's, few and equal values, both peak modes."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _want(S, k, raw):
    F = S.size
    l, r = np.r_[-np.inf, S[:-1]], np.r_[S[1:], -np.inf]
    peak = np.ones(F, bool) if raw or F == 1 else (S > l) & (S >= r)
    if not raw and F > 1:
        peak[0] = S[0] >= S[1]
    e = np.flatnonzero(peak)
    e = e[np.lexsort((e, -S[e].astype(np.float64)))][:k]
    return np.r_[e, np.full(k - e.size, -1)]


@pytest.mark.parametrize("raw", [False, True])
@pytest.mark.parametrize("k", [1, 5, 31, 32, 33, 64])
@pytest.mark.parametrize("F", [1, 2, 33, 128, 129, 2047, 2048, 2049, 5000])
def test_peaks_of_the_dense_values(F, k, raw):
    import paper_2502_00243_gb300 as G

    rng = np.random.default_rng([29, F, k])
    ns = [300, 1, 2, 40]  # one observation: all values equal
    off = np.concatenate([[0], np.cumsum(ns)]).astype(np.int64)
    t, x, s = rng.uniform(0, 500, off[-1]), rng.normal(size=off[-1]), rng.uniform(0.1, 0.4, off[-1])
    d = [torch.from_numpy(v).cuda() for v in (off, t, x, s, 0.5 + np.arange(F) / 4096.0)]
    S = torch.empty(len(ns) * F, dtype=torch.float64, device="cuda")
    idx = torch.full((len(ns) * k,), -9, dtype=torch.int32, device="cuda")
    Sk = torch.zeros(len(ns) * k, dtype=torch.float32, device="cuda")
    p = G.fpw_params_default(peak_mode=G.FPW_PEAK_RAW if raw else G.FPW_PEAK_LOCALMAX)
    G.fpw_periodogram_drift(G.Context(0), None, p, *d, 9, 1, 1.0, k, idx, Sk, S)
    # the peaks rank the FP32 values: the dense ones rounded
    S32 = S.cpu().numpy().astype(np.float32).reshape(len(ns), F)
    idx, Sk = idx.cpu().numpy().reshape(len(ns), k), Sk.cpu().numpy().reshape(len(ns), k)
    for c in range(len(ns)):
        want = _want(S32[c], k, raw)
        assert np.array_equal(idx[c], want)
        assert np.array_equal(Sk[c][want >= 0], S32[c][want[want >= 0]])
        assert np.isnan(Sk[c][want < 0]).all()
