"""Curves at common times in pairs of 64-curve groups (one accumulator a part)
against the same curves in a group by themselves (rows side by side): counts of
curves around 64 and 128, bins around 8 columns and an accumulator's width,
observations around a chunk and around none.

Both multiply the same operands in the same order; the reductions add M terms of
FP32 in different orders, at most M + 8 roundings of 2^-23 of their sum."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [0, 1, 32, 33, 97])
@pytest.mark.parametrize("M", [1, 7, 8, 20, 50, 85, 129, 256])
@pytest.mark.parametrize("C", [65, 128, 129, 200])
def test_pairs_against_single_groups(C, M, n):
    import paper_2502_00243_gb300 as G

    rng = np.random.default_rng([31, C, M, n])
    F, k = 47, 2
    t, f = rng.uniform(-100.0, 700.0, n), 0.125 + np.arange(F) / 4096.0
    x, s = rng.normal(size=(C, n)), rng.uniform(0.02, 0.4, (C, n))
    if n > 0:
        s[5, 0] = 0.0  # a bad curve among good ones

    def run(rows):
        d = [torch.from_numpy(np.ascontiguousarray(v)).cuda() for v in (t, x[rows], s[rows], f)]
        S = torch.full((len(rows) * F,), -1.0, dtype=torch.float64, device="cuda")
        idx = torch.zeros(len(rows) * k, dtype=torch.int32, device="cuda")
        Sk = torch.zeros(len(rows) * k, dtype=torch.float32, device="cuda")
        G.fpw_periodogram_shared(G.Context(0), None, G.fpw_params_default(), *d, M, k, idx, Sk, S)
        return S.cpu().numpy().reshape(len(rows), F)

    got = run(np.arange(C))
    want = np.concatenate([run(np.arange(c, min(c + 64, C))) for c in range(0, C, 64)])
    bad = np.isnan(want)
    assert np.array_equal(np.isnan(got), bad) and (n == 0 or bad[5].all())
    assert (np.abs(got - want)[~bad] <= (M + 8) * 2.0 ** -23 * np.abs(want)[~bad]).all()
