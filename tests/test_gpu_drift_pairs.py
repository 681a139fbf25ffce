"""The drift reduction in FP32 pairs against the one in binary64, on the same bins.

Scaling x, sigma and beta by 2^-20 leaves H0, every phase and, up to an exact
power of two, every bin as they are, and takes the weights out of the pair
reduction's range, so the two dense results are S from equal bins by the two
reductions. A pair carries 2^-46, a frequency adds M bins and a K x K system,
and H0 >= I bounds the condition by its trace."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K", [0, 1, 2, 3, 4])
@pytest.mark.parametrize("M,inv_alpha2", [(1, 0.0), (7, 0.25), (10, 0.0), (20, 0.0), (33, 2.0 ** -40), (50, 0.0)])
def test_pairs_against_binary64(M, inv_alpha2, K):
    import paper_2502_00243_gb300 as G

    rng = np.random.default_rng([23, M, K])
    ns = [1, 2, 5, 119, 120, 121, 240, 700]
    off = np.concatenate([[0], np.cumsum(ns)]).astype(np.int64)
    t = rng.uniform(-50.0, 900.0, off[-1])
    x, s = rng.normal(size=off[-1]) + 3.0, rng.uniform(0.05, 0.5, off[-1])
    F, k, beta = 517, 4, 0.75
    f = 0.25 + np.arange(F) / 8192.0
    out = []
    for scale in (1.0, 2.0 ** -20):
        d = [torch.from_numpy(v).cuda() for v in (off, t, x * scale, s * scale, f)]
        S = torch.full((len(ns) * F,), -1.0, dtype=torch.float64, device="cuda")
        idx = torch.full((len(ns) * k,), -9, dtype=torch.int32, device="cuda")
        Sk = torch.zeros(len(ns) * k, dtype=torch.float32, device="cuda")
        p = G.fpw_params_default(inv_alpha2=inv_alpha2 * scale ** -2)
        G.fpw_periodogram_drift(G.Context(0), None, p, *d, M, K, beta * scale, k, idx, Sk, S)
        out.append((S.cpu().numpy().reshape(len(ns), F), idx.cpu().numpy().reshape(len(ns), k)))
    (Sp, ip), (Sd, id_) = out
    for c in range(len(ns)):
        w = s[off[c]:off[c + 1]] ** -2
        trace = 1.0 + max(K, 1) * (1.0 + beta * beta * w.sum())
        assert np.abs(Sp[c] - Sd[c]).max() <= (M + 16) * 2.0 ** -46 * trace * max(Sd[c].max(), 1e-300)
        # both report peaks; where they differ the two periodograms hold equal values to the same bound
        assert (ip[c] >= 0).sum() == (id_[c] >= 0).sum()
