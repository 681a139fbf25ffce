"""A curve's S at common times is the same bit for bit however the call's groups of
64 curves are taken: pairs and a group left over, with several items per block and
an epilogue behind the next item's first chunk, against each group by itself. The
launch rule is restated here, so a changed rule cannot leave the pairs out."""
from __future__ import annotations

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def pair_groups(groups, F, fpm, nsm):
    paired, single = -(-F // fpm), -(-F // (2 * fpm))

    def rounds(items):
        return -(-items // nsm)
    pairs = 9 * rounds(groups // 2 * paired) + 10 * rounds(groups % 2 * single)
    return groups & ~1 if pairs <= 10 * rounds(groups * single) else 0


@pytest.mark.parametrize("n", [0, 1, 32, 33, 200])
@pytest.mark.parametrize("M", [1, 3, 7, 8, 11, 20, 50, 85, 129, 256])
@pytest.mark.parametrize("C", [128, 185])
def test_pairs_and_a_group_left_over(C, M, n):
    import paper_2502_00243_gb300 as G

    nsm = torch.cuda.get_device_properties(0).multi_processor_count
    fpm = min(64, 256 // M)
    F = 2 * fpm * 2 * nsm - 3  # four passes a block in pairs, two for a group left over
    groups = -(-C // 64)
    assert pair_groups(groups, F, fpm, nsm) == 2
    gen = torch.Generator(device="cuda")
    gen.manual_seed(1000 * M + n)
    x = torch.randn(C, n, generator=gen, device="cuda", dtype=torch.float64)
    s = 0.05 + torch.rand(C, n, generator=gen, device="cuda", dtype=torch.float64)
    t = 700.0 * torch.rand(n, generator=gen, device="cuda", dtype=torch.float64)
    f = 0.125 + torch.arange(F, device="cuda", dtype=torch.float64) / 4096.0
    ctx = G.Context(0)

    def run(c0, c1):
        S = torch.full(((c1 - c0) * F,), -1.0, dtype=torch.float64, device="cuda")
        idx = torch.zeros((c1 - c0) * 3, dtype=torch.int32, device="cuda")
        Sk = torch.zeros((c1 - c0) * 3, dtype=torch.float32, device="cuda")
        G.fpw_periodogram_shared(ctx, None, None, t, x[c0:c1].contiguous(), s[c0:c1].contiguous(), f, M, 3, idx, Sk, S)
        assert ctx.status() == 0
        return S.cpu().numpy(), idx.cpu().numpy(), Sk.cpu().numpy()

    got = run(0, C)
    want = [np.concatenate(q) for q in zip(*[run(c, min(c + 64, C)) for c in range(0, C, 64)])]
    for a, b in zip(got, want):
        np.testing.assert_array_equal(a, b)
