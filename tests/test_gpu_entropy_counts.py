"""The dense phase entropy's counts at the edges of its launches: the number of
bins where a thread's frequencies change, frequency counts on both sides of
where the grid is cut finer, and observation counts around the staged chunk.

Grids are dyadic, so the stepped phases are exact to 2^-54 cycles and no
observation changes bins. The FP32 sum of up to M terms N_m log N_m <= N log N
and the final log N - sum / N carry at most M + 4 roundings of 2^-24 log N."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 7, 255, 256, 257, 513])
@pytest.mark.parametrize("M,F", [(1, 40), (12, 1025), (13, 513), (24, 511), (25, 257), (96, 255), (97, 129), (256, 1)])
def test_counts_at_the_edges(M, F, n):
    _check(M, F, n)


# blocks of 128 R frequencies while at least 304 of them (152 for R = 2): one frequency before and after each change of R
@pytest.mark.parametrize("M,F", [(M, (303 if R > 2 else 151) * 128 * R + d) for M, rs in ((5, (8, 4, 2)), (20, (4, 2)), (50, (2,)))
                                 for R in rs for d in (0, 1)])
def test_counts_where_the_launch_changes(M, F):
    _check(M, F, 9)


def _check(M, F, n):
    import paper_2502_00243_gb300 as G

    rng = np.random.default_rng([17, M, F, n])
    t = rng.uniform(-400.0, 900.0, n)
    freqs = 0.0625 + np.arange(F) / 16384.0
    H = torch.full((F,), -1.0, dtype=torch.float32, device="cuda")
    G.fpw_phase_entropy(G.Context(0), None, torch.from_numpy(t).cuda(), torch.from_numpy(freqs).cuda(), M, H)
    want = oracle.phase_entropy(t, freqs, M)
    assert np.abs(H.cpu().numpy() - want).max() <= (M + 4) * 2.0 ** -24 * max(1.0, np.log(n))
