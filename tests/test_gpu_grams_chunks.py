"""The Grams that create, set_factors and the gradient form: a block's rows pass through shared memory
2048 / R at a time, a thread sums one Gram pair over them, and from rank 24 on (more than 288 pairs)
some threads sum two.  Rows below, at and beyond a chunk at low and high ranks.

Tolerance: FP64 sums of at most 5000 terms, 1e-12 relative to ||T||^2 + ||X||^2."""
import numpy as np
import pytest

from paper_2112_03985_gb300 import api

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,ranks", [((5000, 4, 6), [1, 2, 3]), ((2048, 3, 5), [1]), ((1025, 3, 4), [2, 1]),
                                        ((700, 3, 4), [23, 24, 32, 3]), ((64, 65, 3), [32, 31])],
                         ids=lambda x: "x".join(map(str, x)))
def test_loss_of_given_factors(dims, ranks):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    rng = np.random.default_rng(sum(dims))
    T = rng.standard_normal(dims)
    U = [rng.standard_normal((I, sum(ranks))) for I in dims]
    with api.JKCALS(T, 0, ranks, [[] for _ in ranks], U) as h:
        f, _ = h.grad(want_grad=False)
    offs = np.concatenate([[0], np.cumsum(ranks)])
    want = scale = 0.0
    for a, b in zip(offs[:-1], offs[1:]):
        X = np.einsum("iz,jz,kz->ijk", *[u[:, a:b] for u in U], optimize=True)
        want += np.sum((T - X) ** 2)
        scale += np.sum(T ** 2) + np.sum(X ** 2)
    assert abs(f - want) <= 1e-12 * scale
