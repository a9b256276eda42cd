"""Contractions over a mode of more than 65535 x 8 indices with one or two outputs per row: the
split over the terms meets the limit of the launch grid.  MTTKRPs and a sweep against FP64."""
import numpy as np
import pytest

from paper_2112_03985_gb300 import api

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,ranks", [((4, 1, 600000), [1]), ((4, 1, 524281), [1]), ((4, 1, 600001), [1, 1]),
                                        ((1, 3, 700000), [1])],
                         ids=lambda x: "x".join(map(str, x)))
def test_long_mode(dims, ranks):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    rng = np.random.default_rng(dims[-1])
    T = rng.random(dims)
    U = [rng.random((I, len(ranks))) for I in dims]
    left = [[] for _ in ranks]
    with api.JKCALS(T, 0, ranks, left, U) as h, api.JKCALS(T, 0, ranks, left, U, max_device_bytes=1 << 40) as native:
        for n in range(3):
            others = [U[k] for k in range(3) if k != n]
            letters = "abc"
            spec = "abc," + ",".join(letters[k] + "z" for k in range(3) if k != n) + "->" + letters[n] + "z"
            want = np.einsum(spec, T, *others)
            # sums of at most 2.8e6 positive FP64 terms: 2.8e6 x 2^-53 of the sum bounds both
            np.testing.assert_allclose(np.asarray(h.mttkrp(n)), want, rtol=3e-10)
        h.als_sweep(2), native.als_sweep(2)
        for a, b in zip(h.get_factors(), native.get_factors()):
            np.testing.assert_allclose(np.asarray(a), np.asarray(b), rtol=1e-8)
