"""The exact-chain form's slicing of the tensor: entries of at most 24 significant bits are cut in
FP32, the others in FP64, and both must give the same slices.  The same tensor with every entry
moved by 2^-40 of itself takes the other branch; its slices may differ by one unit of the last one
(2^-28 of a row's largest entry), so the MTTKRPs agree within the form's bar of 1e-8."""
import numpy as np
import pytest

from paper_2112_03985_gb300 import api

from _helpers import assert_elementwise

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scale", [0, -100, 100], ids=lambda s: f"2^{s}")
@pytest.mark.parametrize("dims", [(33, 20, 17), (9, 150, 30)], ids=lambda d: "x".join(map(str, d)))
def test_both_slicings_agree(dims, scale):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    rng = np.random.default_rng(sum(dims))
    T = rng.random(dims).astype(np.float32).astype(np.float64)
    T[rng.random(dims) < 0.1] = 0.0
    T[0] *= 2.0 ** -20                       # small against the rows they share
    T = np.ldexp(T, scale)
    ranks = [4] * 9
    U = [rng.random((I, sum(ranks))) for I in dims]
    left = [[] for _ in ranks]
    with api.JKCALS(T, 0, ranks, left, U, precision="exact_bf16") as a, \
            api.JKCALS(T * (1 + 2.0 ** -40), 0, ranks, left, U, precision="exact_bf16") as b:
        for n in range(3):
            x, y = np.asarray(a.mttkrp(n)), np.asarray(b.mttkrp(n))
            for i in range(x.shape[0]):
                assert_elementwise(x[i], y[i], 1e-8, f"mode {n} row {i}")
