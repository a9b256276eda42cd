"""The FP64 form's tensor-times-matrix route (BF16 digits on the tensor cores, one product shared
by several modes) against plain FP64 arithmetic and against the CUDA-core kernel, at the edges of
its tiles: contractions around a multiple of 16, around the tile widths' border and at their
longest, columns around a multiple of 128, rows around a multiple of 32 and 64, 2 to 5 modes,
non-finite and widely scaled inputs.

Tolerance: both routes sum at most 1.2e5 FP64 terms, whose rounding is far below the FP64 form's
MTTKRP bar of 1e-12 of the largest entry; the digits drop less than one FP64 rounding per term."""
import numpy as np
import pytest

from paper_2112_03985_gb300 import api

from _helpers import assert_elementwise

pytestmark = pytest.mark.gpu

BAR = 1e-12


def _torch():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch


def _inputs(dims, ranks, seed, positive=False):
    rng = np.random.default_rng(seed)
    draw = rng.random if positive else (lambda s: rng.standard_normal(s))
    return draw(dims), [draw((I, sum(ranks))) for I in dims]


def _reference(T, U, n):
    """Mode n's MTTKRP by einsum in FP64."""
    letters = "abcdefgh"[:T.ndim]
    args = [letters + "," + ",".join(letters[k] + "z" for k in range(T.ndim) if k != n) + "->" + letters[n] + "z"]
    return np.einsum(args[0], T, *[U[k] for k in range(T.ndim) if k != n], optimize=True)


def _handles(T, ranks, U, **kw):
    """The same problem on the planned route and on the CUDA-core kernel (a memory cap, here one
    that nothing reaches, keeps a handle on it, with the plan it would have without the route)."""
    left = [[] for _ in ranks]
    return (api.JKCALS(T, 0, ranks, left, U, **kw),
            api.JKCALS(T, 0, ranks, left, U, max_device_bytes=1 << 46, **kw))


def _assert_routes_differ(h, native):
    """The same sums in another order: after a sweep some factor differs in its last bits."""
    assert any((np.asarray(a) != np.asarray(b)).any() for a, b in zip(h.get_factors(), native.get_factors())), \
        "this size does not take the route under test"


SHAPES = [   # dims, ranks
    ((48, 65, 63), [4] * 32),               # C = 128, one tile each way and one row more
    ((47, 64, 129), [3] * 43),              # C = 129
    ((33, 49, 80), [1, 2, 3, 4, 7] * 20),   # mixed ranks
    ((448, 40, 37), [5] * 60),              # the longest exact chain
    ((449, 40, 37), [5] * 60),              # one longer: that mode is never contracted
    ((176, 177, 21), [5] * 77),             # the tile widths' two sides
    ((300, 500), [6] * 200),                # two modes: the product is the MTTKRP
    ((61, 40, 50), [3] * 171),              # odd C: single-column loads
    ((30, 17, 25, 31), [8] * 50),
    ((12, 13, 9, 11, 14), [6] * 80),
]


@pytest.mark.parametrize("dims,ranks", SHAPES, ids=["x".join(map(str, s[0])) for s in SHAPES])
def test_mttkrps_sweep_and_gradient(dims, ranks):
    _torch()
    T, U = _inputs(dims, ranks, seed=sum(dims))
    h, native = _handles(T, ranks, U)
    with h, native:
        refs = [_reference(T, U, n) for n in range(len(dims))]
        for n, ref in enumerate(refs):
            assert_elementwise(h.mttkrp(n), ref, BAR, f"mode {n}")
        (f0, G0), (f1, G1) = h.grad(), native.grad()
        assert abs(f0 - f1) <= 1e-12 * abs(f1)
        # G = 2 (U H - M): the MTTKRP's bar against the larger of both terms
        for n, (a, b) in enumerate(zip(G0, G1)):
            scale = max(np.abs(b).max(), 2 * np.abs(refs[n]).max())
            assert np.abs(np.asarray(a) - np.asarray(b)).max() <= 4 * BAR * scale, n
        h.als_sweep(1), native.als_sweep(1)
        _assert_routes_differ(h, native)


def test_sweeps_match_the_cuda_core_route():
    _torch()
    T, U = _inputs((40, 33, 61), [5] * 41, seed=3, positive=True)
    h, native = _handles(T, [5] * 41, U)
    with h, native:
        la, lb = h.als_sweep(6), native.als_sweep(6)
        np.testing.assert_allclose(la, lb, rtol=1e-10)
        for a, b in zip(h.get_factors(), native.get_factors()):
            assert_elementwise(a, b, 1e-10)


def test_scaled_slices_and_exact_values():
    """Slices and columns of very different magnitudes keep their relative accuracy, and small
    integers (every digit sum exact, level sums up to the chain bound) come out exactly."""
    _torch()
    dims, ranks = (448, 30, 40), [5] * 60
    rng = np.random.default_rng(5)
    T, U = _inputs(dims, ranks, seed=6)
    T *= 10.0 ** rng.integers(-120, 120, (448, 1, 1))     # an outlying sample per slice
    for u in U:
        u *= 10.0 ** rng.integers(-20, 20, (1, u.shape[1]))
    keep = rng.random(U[0].shape) < 0.5
    U[0] = np.where(keep, U[0], 0.0)
    h, native = _handles(T, ranks, U)
    with h, native:
        for n in (1, 2):
            a, b = np.asarray(h.mttkrp(n)), np.asarray(native.mttkrp(n))
            for c in range(a.shape[1]):
                assert_elementwise(a[:, c], b[:, c], BAR, f"mode {n} column {c}")
    T = np.full(dims, 127.0)
    U = [np.full((I, sum(ranks)), 127.0) for I in dims]
    T[::2] = -127.0
    T[:, ::3] = 127.0
    h, native = _handles(T, ranks, U)
    with h, native:
        for n in range(3):
            np.testing.assert_array_equal(h.mttkrp(n), _reference(T, U, n))


@pytest.mark.parametrize("value", [np.inf, -np.inf, np.nan, 1e308, 5e-324])
def test_non_finite_and_extreme_values(value):
    """A factor entry that is Inf, NaN, huge or subnormal gives what the CUDA-core kernel gives;
    so does a tensor entry."""
    _torch()
    dims, ranks = (40, 33, 61), [5] * 41
    for where in ("factor", "tensor"):
        T, U = _inputs(dims, ranks, seed=7, positive=True)
        if where == "factor":
            for n, u in enumerate(U):
                u[3 + n, 10 + 7 * n] = value
        else:
            T[5, 6, 7] = value
        h, native = _handles(T, ranks, U)
        with h, native:
            for n in range(3):
                a, b = np.asarray(h.mttkrp(n)), np.asarray(native.mttkrp(n))
                fin = np.isfinite(b)
                np.testing.assert_array_equal(a[~fin], b[~fin])
                for c in range(a.shape[1]):
                    if fin[:, c].all():
                        assert_elementwise(a[:, c], b[:, c], BAR, f"{where} mode {n} column {c}")
