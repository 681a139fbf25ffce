"""Whether phases step along the grid's line is decided for all frequencies
between two anchors, whichever part of them a block or a pass holds: a call with
few frequencies or in pairs of groups takes the same bins as any other.

The grid lies on a line but for two frequencies of one span. One is 1e-13 below
it (1e-10 cycles at t = 1024: within the tolerance), where an observation's phase
on the line is a whole number, so its bin is the last one by the exact phase and
the first one by the step. The other is far off the line, so all of the span's
phases are exact. H is that of the exact bins to 1e-5 (0 with the
other ones), S to 1e-5 of the sum of w x^2 (FP32 bin sums of 63 observations)."""
from __future__ import annotations

import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def grid(F, below, off):
    f = 1.0 + np.arange(F) / 1024.0
    f[below] -= 1e-13
    f[off] += 1e-5
    return f


@pytest.mark.parametrize("M,span", [(10, 1024), (20, 512), (50, 256), (97, 128)])
@pytest.mark.parametrize("spans", [1, 2, 700])
def test_entropy(M, span, spans):
    import paper_2502_00243_gb300 as G

    F = span * spans - 1
    f = grid(F, 5, span - 3)
    t = np.array([1024.0, 1024.0, 1024.0, 0.0, 0.0])
    H = torch.full((F,), -1.0, dtype=torch.float32, device="cuda")
    G.fpw_phase_entropy(G.Context(0), None, torch.from_numpy(t).cuda(), torch.from_numpy(f).cuda(), M, H)
    want = oracle.phase_entropy(t, f, M)
    assert want[5] > 0.5
    assert abs(float(H[5]) - want[5]) < 1e-5


@pytest.mark.parametrize("M", [5, 20, 50])
@pytest.mark.parametrize("C", [64, 128, 256])
def test_common_times(C, M):
    import paper_2502_00243_gb300 as G

    fpm = min(64, 256 // M)
    F = 6 * fpm - 1
    f = grid(F, 1, 2 * fpm - 1)
    rng = np.random.default_rng([5, C, M])
    t = np.concatenate([np.full(3, 1024.0), rng.integers(0, 1024, 60) / 7.0])
    x, s = rng.normal(size=(C, t.size)), rng.uniform(0.1, 0.2, (C, t.size))
    d = [torch.from_numpy(v).cuda() for v in (t, x, s, f)]
    S = torch.zeros(C * F, dtype=torch.float64, device="cuda")
    G.fpw_periodogram_shared(G.Context(0), None, None, *d, M, 0, None, None, S)
    got = S.cpu().numpy().reshape(C, F)[:, 1]
    want = np.array([oracle.fpw(t, x[c], s[c], f[1:2], M)[0] for c in range(C)])
    on_line = np.array([oracle.fpw(t, x[c], s[c], f[1:2] + 1e-13, M)[0] for c in range(C)])
    tol = 1e-5 * np.sum(x * x / (s * s), axis=1)
    assert (np.abs(want - on_line) > 10.0 * tol).sum() > C // 2
    assert (np.abs(got - want) <= tol).all()
