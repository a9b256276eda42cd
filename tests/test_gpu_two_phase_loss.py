"""The order of the two-phase update's loss: the H * G term is summed by 128 threads (entry p of the
R x R products on thread p mod 128, in increasing p, then a tree), whatever the number of threads
that the rest of the kernel uses.  An integer problem whose factors are found exactly makes these
sums the only rounding, so the loss must equal the same additions done here, bit for bit."""
import numpy as np
import pytest

from paper_2112_03985_gb300 import api

pytestmark = pytest.mark.gpu


def _tree(x):
    x = x.copy()
    w = len(x) // 2
    while w > 0:
        x[:w] += x[w:2 * w]
        w //= 2
    return x[0]


def _sums(H, G, V, M, threads):
    """sum(H * G) and sum(V * M) in the kernels' order; multiply-adds round once."""
    R = len(H)
    part = np.zeros(threads)
    for p in range(R * R):
        part[p % threads] = float(int(part[p % threads]) + int(H[p // R, p % R]) * int(G[p // R, p % R]))
    rows = np.zeros(128)
    for i in range(R):
        for r in range(R):
            rows[i] = float(int(rows[i]) + int(V[i, r]) * int(M[i, r]))
    return _tree(part), _tree(rows)


@pytest.mark.parametrize("R,seed", [(12, 131), (16, 6), (20, 9), (32, 3), (32, 5)])
def test_loss_bits(R, seed):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    rng = np.random.default_rng(seed)

    def factor():   # unit upper triangular, its Gram's Cholesky factor its own transpose
        X = np.eye(R, dtype=np.int64)
        X[0, 1:] = rng.integers(4096, 16384, R - 1)
        return X

    A, V = factor(), factor()
    T, H, G = A @ V.T, A.T @ A, V.T @ V
    hg, fit = _sums(H, G, V, V @ H, 128)
    assert hg != _sums(H, G, V, V @ H, 512)[0]      # the case tells the orders apart
    with api.JKCALS(T.astype(float), 0, [R], [[]], [np.ones((R, R)), V.astype(float)], normalise=False,
                    update_mode=2) as h:
        nt, _ = h.grad(U=[np.zeros((R, R))] * 2, want_grad=False)
        got = np.asarray(h.als_sweep(1))[0, 0]
        U = h.get_factors()
    np.testing.assert_array_equal(U[0], A)
    np.testing.assert_array_equal(U[1], V)
    assert got == nt + hg - 2.0 * fit
