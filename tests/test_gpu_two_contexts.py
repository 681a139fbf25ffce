"""Calls of different sizes from two threads, each with a context of its own: both
take the same kernel at different bin counts, so the blocks differ in shared memory,
and the limit that one of them sets must do for the other."""
from __future__ import annotations

import threading

import pytest

import lightcurves as L
from gpu_util import to_dev

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("call", ["batch", "noalloc", "entropy", "entropy_peaks"])
def test_two_contexts_at_different_bin_counts(call):
    import paper_2502_00243_gb300 as G

    w = L.ragged(5, [40, 33], 300, M=20, k=2)
    d = to_dev(w)
    p = G.fpw_params_default(threads=128, freqs_per_thread=2)
    errors, start = [], threading.Barrier(2, timeout=60)
    bins = {"entropy": (97, 250), "entropy_peaks": (64, 4096)}.get(call, (5, 50))

    def work(M):
        try:
            ctx, st = G.Context(0), torch.cuda.Stream()
            idx, S = torch.zeros(4, dtype=torch.int32, device="cuda"), torch.zeros(4, dtype=torch.float32, device="cuda")
            H, z = torch.zeros(300, dtype=torch.float32, device="cuda"), torch.zeros(4, dtype=torch.float32, device="cuda")
            torch.cuda.synchronize()
            start.wait()
            for _ in range(2000):
                # (one call at a time without allocation: they share their scratch)
                if call == "batch" or (call == "noalloc" and M == 5):
                    G.fpw_periodogram_batch_ex(ctx, st, p, d["offsets"], w.offsets, d["t"], d["x"], d["sigma"],
                                               d["freqs"], M, 2, idx, S)
                elif call == "noalloc":
                    G.fpw_periodogram_batch_noalloc(st, p, d["offsets"], w.offsets, d["t"],
                                                    d["x"], d["sigma"], d["freqs"], M, 2, idx, S)
                elif call == "entropy":
                    G.fpw_phase_entropy(ctx, st, d["t"], d["freqs"], M, H)
                else:
                    G.fpw_phase_entropy_peaks(ctx, st, d["offsets"], d["t"], d["freqs"], M, 2, idx, H[:4], z)
            st.synchronize()
        except Exception as e:  # noqa: BLE001
            errors.append((M, e))

    threads = [threading.Thread(target=work, args=(M,)) for M in bins]
    for th in threads:
        th.start()
    for th in threads:
        th.join()
    torch.cuda.synchronize()
    assert not errors, errors
