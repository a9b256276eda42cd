"""The exact-chain form's slicing of a tensor whose padded unfolding has more than 2^31 entries (64-bit
indices): two modes of size 1 are padded 32 rows by 8 columns, so a tensor of 8.4e6 entries is
enough.  MTTKRPs against FP64 within the form's bar of 1e-8."""
import numpy as np
import pytest

from paper_2112_03985_gb300 import api

pytestmark = pytest.mark.gpu


def test_padded_unfolding_beyond_32_bits():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    dims = (2, 1, 1, 4194400)                 # mode 1: 32 x 16 x 4194400 padded entries
    assert 32 * 16 * dims[3] > 2 ** 31
    rng = np.random.default_rng(4)
    T = rng.random(dims)
    U = [rng.random((I, 2)) for I in dims]
    # splits: the planned ones (a chain of columns per CTA) would pass the launch grid
    with api.JKCALS(T, 0, [1, 1], [[], []], U, precision="exact_bf16", splits=152) as h:
        for n in (1, 0, 3):
            got = np.asarray(h.mttkrp(n))
            others = [U[k] for k in range(4) if k != n]
            letters = "abcd"
            spec = "abcd," + ",".join(letters[k] + "z" for k in range(4) if k != n) + "->" + letters[n] + "z"
            want = np.einsum(spec, T, *others)
            np.testing.assert_allclose(got, want, rtol=1e-8, atol=1e-8 * np.abs(want).max())
