"""autotune of an FP64 handle whose sweeps take the shared products: the CUDA-core kernel that single
MTTKRPs, compacted runs and modes without images still run is tuned as on a handle without
them, and the handle goes on with the products."""
import numpy as np
import pytest

from paper_2112_03985_gb300 import api

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,ranks", [((40, 33, 61), [5] * 41), ((120, 64, 64), [4] * 32)],
                         ids=lambda x: "x".join(map(str, x))[:12])
def test_cuda_core_splits_are_tuned(dims, ranks):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    rng = np.random.default_rng(sum(dims))
    T, left = rng.random(dims), [[] for _ in ranks]
    U = [rng.random((I, sum(ranks))) for I in dims]
    with api.JKCALS(T, 0, ranks, left, U) as plain, api.JKCALS(T, 0, ranks, left, U, autotune=True) as tuned:
        (kernels, planned), (tuned_kernels, found) = plain.sweep_info(), tuned.sweep_info()
        # in every mode of both sizes the timing settles on other split factors than the planned ones
        assert found != planned
        assert tuned_kernels == kernels
        plain.als_sweep(3), tuned.als_sweep(3)
        for a, b in zip(plain.get_factors(), tuned.get_factors()):
            np.testing.assert_array_equal(a, b)      # the products' sweeps: the same bits
