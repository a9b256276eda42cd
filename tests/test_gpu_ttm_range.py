"""Entries of very different size in the FP64 form's tensor-times-matrix route: an outlying sample
that submodels leave out, a spike in a single entry, factor columns with a localised large entry
where the tensor is small or zero, noise-free bumps whose tails lie 1e-20 below their peaks, and
sparse tensors.  Every entry of an MTTKRP is held to its own terms: an FP64 sum of J terms is
within J 2^-53 of the sum A of their magnitudes, so two of them (J <= 5000) agree within
1e-12 A, entry by entry."""
import numpy as np
import pytest

from paper_2112_03985_gb300 import api

pytestmark = pytest.mark.gpu

BAR = 1e-12


@pytest.fixture(autouse=True)
def _gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _mttkrp(T, U, n):
    letters = "abcdefgh"[:T.ndim]
    spec = letters + "," + ",".join(letters[k] + "z" for k in range(T.ndim) if k != n) + "->" + letters[n] + "z"
    return np.einsum(spec, T, *[U[k] for k in range(T.ndim) if k != n], optimize=True)


def _handles(T, left, ranks, U):
    """The planned route and the CUDA-core kernel (a memory cap that nothing reaches keeps a
    handle on it)."""
    return api.JKCALS(T, 0, ranks, left, U), api.JKCALS(T, 0, ranks, left, U, max_device_bytes=1 << 46)


def _loo(I, R):
    return [[p] for p in range(I)], [R] * I


def _zeroed(U, left, ranks):
    """The multi-matrices with every block's left-out rows of mode 0 zero."""
    offs = np.concatenate([[0], np.cumsum(ranks)])
    U = [u.copy() for u in U]
    for g, D in enumerate(left):
        U[0][D, offs[g]:offs[g + 1]] = 0.0
    return U


def _check(T, left, ranks, U):
    """MTTKRPs against einsum, entry by entry, on a size that takes the route under test."""
    Z = _zeroed(U, left, ranks)
    h, native = _handles(T, left, ranks, U)
    with h, native:
        for n in range(T.ndim):
            got, ref = np.asarray(h.mttkrp(n)), _mttkrp(T, Z, n)
            A = _mttkrp(np.abs(T), [np.abs(u) for u in Z], n)
            bad = ~(np.abs(got - ref) <= BAR * A)
            assert not bad.any(), f"mode {n}: {bad.sum()} entries, worst {np.nanmax(np.abs(got - ref)[bad] / A[bad]):.1e}"
        h.als_sweep(1), native.als_sweep(1)
        assert any((np.asarray(a) != np.asarray(b)).any() for a, b in zip(h.get_factors(), native.get_factors()))


@pytest.mark.parametrize("size", [1e6, 1e8, 1e12, 1e20])
def test_spike_in_one_sample(size):
    dims = (40, 33, 61)
    rng = np.random.default_rng(11)
    T = rng.random(dims)
    T[5, 6, 7] = size
    left, ranks = _loo(40, 5)
    U = [rng.random((I, sum(ranks))) for I in dims]
    _check(T, left, ranks, U)


def test_factors_of_the_submodel_without_the_spike():
    """The submodel that leaves the outlying sample out is the model of an ordinary tensor (those that
    keep it solve with matrices of condition 1e8 and more, where plain FP64 is 1e-7 off itself)."""
    dims = (40, 33, 61)
    rng = np.random.default_rng(12)
    T = rng.random(dims)
    T[5, 6, 7] = 1e20
    left, ranks = _loo(40, 5)
    U = [rng.random((I, sum(ranks))) for I in dims]
    h, native = _handles(T, left, ranks, U)
    with h, native:
        h.als_sweep(1), native.als_sweep(1)
        for a, b in zip(h.get_factors(), native.get_factors()):
            a, b = np.asarray(a)[:, 25:30], np.asarray(b)[:, 25:30]
            assert np.linalg.norm(a - b) <= 1e-10 * np.linalg.norm(b)


@pytest.mark.parametrize("size", [1e6, 1e20])
def test_outlying_sample(size):
    dims = (40, 33, 61)
    rng = np.random.default_rng(13)
    T = rng.standard_normal(dims)
    T[5] *= size
    left, ranks = _loo(40, 5)
    _check(T, left, ranks, [rng.random((I, sum(ranks))) for I in dims])


@pytest.mark.parametrize("slab", [0.0, 1e-18])
def test_localised_factor_entry_where_the_tensor_is_small(slab):
    dims = (40, 33, 61)
    rng = np.random.default_rng(14)
    T = rng.random(dims)
    T[3, :, ::2], T[:, 9, 1::2], T[::3, :, 17] = slab, slab, slab
    left, ranks = _loo(40, 5)
    U = [rng.random((I, sum(ranks))) for I in dims]
    U[0][3, ::2], U[1][9, 1::2], U[2][17, ::3] = 1e9, 1e18, 1e14
    _check(T, left, ranks, U)


@pytest.mark.parametrize("dims", [(40, 100, 50), (40, 50, 34, 20)], ids=lambda d: "x".join(map(str, d)))
def test_noise_free_bumps(dims):
    rng = np.random.default_rng(15)
    left, ranks = _loo(40, 3)
    F = [np.exp(0.5 * rng.standard_normal((dims[0], 3)))]
    for I in dims[1:]:
        x, mu = np.arange(I)[:, None], I * (0.2 + 0.3 * np.arange(3))[None, :]
        F.append(np.exp(-((x - mu) ** 2) / (2 * (0.06 * I) ** 2)))
    letters = "abcd"[:len(dims)]
    T = np.einsum(",".join(l + "z" for l in letters) + "->" + letters, *F)
    U = [np.tile(f, (1, 40)) for f in F]
    _check(T, left, ranks, U)


@pytest.mark.parametrize("density", [0.3, 0.02])
def test_sparse_tensor(density):
    dims = (40, 33, 61)
    rng = np.random.default_rng(16)
    T = np.where(rng.random(dims) < density, rng.integers(1, 50, dims).astype(float), 0.0)
    T[7] = 0.0
    T[:, 8, :] = 0.0
    left, ranks = _loo(40, 5)
    U = [rng.standard_normal((I, sum(ranks))) for I in dims]
    U[1][:, 3] = 0.0
    _check(T, left, ranks, U)


@pytest.mark.parametrize("dims", [(40, 33, 61), (30, 17, 25, 31)], ids=lambda d: "x".join(map(str, d)))
@pytest.mark.parametrize("power", [1, -1])
def test_products_beyond_the_range_that_another_factor_brings_back(dims, power):
    """T times one factor leaves FP64's range, the Khatri-Rao product of the factors does not."""
    rng = np.random.default_rng(17)
    ranks = [5] * 41
    left = [[] for _ in ranks]
    T = rng.standard_normal(dims)
    U = [rng.standard_normal((I, sum(ranks))) for I in dims]
    T[3, 4, 5] = 1e9
    U[1][4, ::7] = 0.0   # entries of every kind: by digits and as plain sums
    refs = [_mttkrp(T, U, n) for n in range(len(dims))]
    bars = [BAR * _mttkrp(np.abs(T), [np.abs(u) for u in U], n) for n in range(len(dims))]
    for big in range(len(dims)):
        for small in range(len(dims)):
            if big == small:
                continue
            V = [u.copy() for u in U]
            V[big] = np.ldexp(U[big], 560 * power)
            V[small] = np.ldexp(U[small], -700 * power)
            S = np.ldexp(T, 480 * power)
            h, native = _handles(S, left, ranks, V)
            with h, native:
                for n in range(len(dims)):
                    if n in (big, small):
                        continue
                    for x in (native, h):
                        got = np.ldexp(np.asarray(x.mttkrp(n)), -340 * power)
                        assert (np.abs(got - refs[n]) <= bars[n]).all(), (big, small, n)
