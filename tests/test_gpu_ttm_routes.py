"""FP64 handles on the shared products in the calls that change or share their route: branches of a
batch, a run whose compaction crosses to the CUDA-core kernel, and digit sums at the chain bound."""
from fractions import Fraction

import numpy as np
import pytest

from paper_2112_03985_gb300 import api, workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _on_products(T, ranks, U, n):
    """Whether mode n's MTTKRP of these inputs is not the CUDA-core kernel's."""
    left = [[] for _ in ranks]
    with api.JKCALS(T, 0, ranks, left, U) as h, api.JKCALS(T, 0, ranks, left, U, max_device_bytes=1 << 46) as native:
        return (np.asarray(h.mttkrp(n)) != np.asarray(native.mttkrp(n))).any()


def test_batched_handles_equal_individual_sweeps():
    ws = [W.make_workload(f"b{k}", dims, R, blocks=W.loo_blocks(dims[0], include_full=True), noise=0.01, seed=80 + k)
          for k, (dims, R) in enumerate([((40, 33, 61), 5), ((48, 64, 40), 4), ((30, 17, 25, 31), 8)])]
    assert all(_on_products(w.T, w.ranks, api.multi_init(w.init), 0) for w in ws)
    hs_a, hs_b = ([api.from_workload(w) for w in ws] for _ in range(2))
    try:
        ref = [(h.als_sweep(7), h.get_factors()) for h in hs_a]
        with api.Batch(hs_b, max_sweeps=4) as b:
            first = []
            for n in (4, 3):
                b.sweep(n)
                b.sync()
                first.append([h.loss_history(n) for h in hs_b])
            got = [(np.concatenate([x[k] for x in first]), h.get_factors()) for k, h in enumerate(hs_b)]
        for (la, Ua), (lb, Ub) in zip(ref, got):
            np.testing.assert_array_equal(la, lb)
            for x, y in zip(Ua, Ub):
                np.testing.assert_array_equal(x, y)
    finally:
        for h in hs_a + hs_b:
            h.close()


def test_compaction_crosses_to_the_cuda_core_kernel():
    """576 columns take the products, the last active blocks the CUDA-core kernel; every block stops
    at the same sweep as without compaction.  Both routes round FP64 sums, 1e-15 a sweep: at most
    400 sweeps of systems of condition 1e4 keep them within 1e-8."""
    blocks, ranks = W.all_ranks_blocks(24, (3, 5, 7, 9))
    w = W.make_workload("all 24x31x40 R3-9", (24, 31, 40), 7, blocks=blocks, ranks=ranks, noise=0.01, seed=71)
    U = api.multi_init(w.init)
    assert _on_products(w.T, w.ranks, U, 1)
    res = {}
    for compact in (True, False):
        with api.from_workload(w, compact=compact) as h:
            done, final = h.run(400, tol=1e-7)
            res[compact] = (done, final, h.run_block_sweeps(), h.block_status(), h.get_factors())
            again = h.als_sweep(2)         # back on the products in the full layout
            assert again.shape == (2, w.K)
    (d1, f1, p1, s1, U1), (d0, f0, p0, s0, U0) = res[True], res[False]
    late = int(sum(np.asarray(w.ranks)[p1 > d1 - 16]))
    assert late <= 64, "the last sweeps run few enough columns for the CUDA-core kernel"
    np.testing.assert_array_equal(p1, p0)
    np.testing.assert_array_equal(s1, s0)
    assert d1 == d0
    np.testing.assert_allclose(f1, f0, rtol=1e-8)
    for a, b in zip(U1, U0):
        np.testing.assert_allclose(a, b, rtol=1e-8, atol=1e-8 * np.abs(b).max())


def _value(d0, d):
    """d0 + sum_{k=1..6} d 2^-7k: balanced digits d0, d, ..., d (50 bits)."""
    return d0 + sum(d * 2.0 ** (-7 * k) for k in range(1, 7))


@pytest.mark.parametrize("K,C", [(448, 600), (102, 900), (103, 900)])
def test_level_sums_at_the_chain_bound(K, C):
    """Every digit at its largest and of one sign: the level sums reach (l + 3) 2^12 K, for K = 448
    within 2% of FP32's 2^24, and K = 102, 103 are the drain's two conversions.  The two-mode
    product is the MTTKRP; one rounding and the dropped products are within 2^-52 of each entry."""
    dims = (K, 448)
    x = np.array([_value(127, 63), -_value(127, 64), _value(64, 63), _value(-127, 63), _value(1, -64)])
    assert abs(x).max() < 128
    T = np.broadcast_to(x[np.arange(448) % 5], dims).copy()
    U = [np.broadcast_to(x[np.arange(C) % 5], (I, C)).copy() for I in dims]
    ranks = [1] * C
    assert _on_products(np.random.default_rng(0).random(dims), ranks, [np.random.default_rng(1).random((I, C)) for I in dims], 1)
    with api.JKCALS(T, 0, ranks, [[] for _ in ranks], U) as h:
        got = np.asarray(h.mttkrp(1))
    for j in range(5):
        for c in range(5):
            want = Fraction(x[j]) * Fraction(x[c]) * K
            block = got[j::5, c::5]
            assert (block == block[0, 0]).all()
            assert abs(Fraction(float(block[0, 0])) - want) <= abs(want) / 2 ** 52, (j, c)
