"""Grouped batches whose problems mix ranks 9 to 12, the class between 8 and 16 of the update's
compile-time sizes: every problem's sweep as its own handle computes it, bit for bit."""
import numpy as np
import pytest

from paper_2112_03985_gb300 import api, workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["3xtf32", "exact_bf16"])
@pytest.mark.parametrize("top", [9, 12])
def test_mixed_ranks(top, precision):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    ws = []
    for k, dims in enumerate([(20, 36, 50), (13, 60, 33)]):
        blocks, ranks = W.all_ranks_blocks(dims[0], (2, 7, top))
        ws.append(W.make_workload(f"r{top} {k}", dims, top, blocks=blocks, ranks=ranks, noise=0.01, seed=90 + k))
    hs_a, hs_b = ([api.from_workload(w, precision=precision) for w in ws] for _ in range(2))
    try:
        ref = [(h.als_sweep(4), h.get_factors()) for h in hs_a]
        with api.Batch(hs_b, max_sweeps=4) as b:
            b.sweep(4)
            b.sync()
            got = [(h.loss_history(4), h.get_factors()) for h in hs_b]
        for (la, Ua), (lb, Ub) in zip(ref, got):
            np.testing.assert_array_equal(la, lb)
            for x, y in zip(Ua, Ub):
                np.testing.assert_array_equal(x, y)
    finally:
        for h in hs_a + hs_b:
            h.close()
