"""The Grams that create, set_factors and the gradient form, at the edges of the kernel's split of a
block over pairs and rows (ranks around 22, where a block's pairs outnumber half its threads, and 32,
where they take two trips; fewer rows than row groups).  The loss of factors is formed from them
alone besides the last mode's MTTKRP, and one sweep's factors solve with them.

Tolerance: FP64 sums of at most a few hundred terms, 1e-12 relative to ||T||^2 + ||X||^2."""
import numpy as np
import pytest

from paper_2112_03985_gb300 import api

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims", [(2, 3, 5), (9, 40, 7), (301, 4, 6)], ids=lambda d: "x".join(map(str, d)))
def test_loss_of_given_factors(dims):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    rng = np.random.default_rng(sum(dims))
    ranks = [1, 2, 22, 23, 31, 32]
    T = rng.standard_normal(dims)
    U = [rng.standard_normal((I, sum(ranks))) for I in dims]
    with api.JKCALS(T, 0, ranks, [[] for _ in ranks], U) as h:
        f, _ = h.grad(want_grad=False)
    offs = np.concatenate([[0], np.cumsum(ranks)])
    want = scale = 0.0
    for a, b in zip(offs[:-1], offs[1:]):
        X = np.einsum("iz,jz,kz->ijk", *[u[:, a:b] for u in U])
        want += np.sum((T - X) ** 2)
        scale += np.sum(T ** 2) + np.sum(X ** 2)
    assert abs(f - want) <= 1e-12 * scale
