"""The FP64 basis products where their integers end: sums that need more than 64 bits, exponents beyond the fixed point
(NaN), and values far below their block's largest.  The products are called directly, by the library's C++ names."""
import ctypes
import math

import numpy as np
import pytest

from paper_0901_3512_gb300 import seedcg
from tests.gpu_helpers import dev, host, need_gpu

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
N = 96                                   # entries: six blocks of 16


def _call(name, *args):
    f = getattr(seedcg.load(), name)
    f.restype = None
    f(*[ctypes.c_void_p(a.data_ptr()) if torch.is_tensor(a) else a for a in args], None)
    torch.cuda.synchronize()


def _gemm(V, runE, coef):
    """Y[j] = sum_a V[a] coef[a][j]"""
    m, nb = coef.shape
    y = torch.zeros(nb, N, dtype=torch.complex128, device="cuda")
    L, I = ctypes.c_long, ctypes.c_int
    _call("_ZN6seedcg10gemm_n_fixEPK7double2liPKiS2_iiPS0_llP11CUstream_st", dev(V), L(N), I(m), dev(runE), dev(coef),
          I(nb), I(nb), y, L(N), L(N))
    return host(y)


def _proj(V, runE, X):
    """C[a][j] = sum_e conj(V[a][e]) X[j][e]"""
    m, n, nx = V.shape[0], V.shape[1], X.shape[0]
    c = torch.zeros(m, nx, dtype=torch.complex128, device="cuda")
    scratch = torch.zeros(1 << 20, dtype=torch.complex128, device="cuda")
    L, I = ctypes.c_long, ctypes.c_int
    _call("_ZN6seedcg8proj_fixEPK7double2liPKiS2_lilPS0_iS5_mP11CUstream_st", dev(V), L(n), I(m), dev(runE), dev(X), L(n),
          I(nx), L(n), c, I(nx), scratch, ctypes.c_size_t(1 << 20))
    return host(c)


def _exponents(V):
    m = np.abs(np.stack([V.real, V.imag])).max(axis=(0, 1)).reshape(-1, 16).max(axis=1)
    return (np.frexp(m)[1] + 1022).astype(np.int32)


@pytest.mark.parametrize("rows", [1, 32, 33, 64, 129, 1000, 5000])
@pytest.mark.parametrize("sign", [1.0, -1.0])
def test_sums_past_64_bits(rows, sign):
    """Products of one sign, all near the largest: 2^56 each in the sums' unit.  Bar: a product is cut at 2^-57 of the
    largest (four of them to a complex one), the sum rounded twice."""
    need_gpu()
    rng = np.random.default_rng(rows)
    V = (rng.uniform(0.9, 0.999, (rows, N)) + 1j * rng.uniform(0.9, 0.999, (rows, N)))
    coef = sign * (rng.uniform(0.9, 0.999, (rows, 3)) - 1j * rng.uniform(0.9, 0.999, (rows, 3)))
    got = _gemm(V, _exponents(V), coef)
    for j in range(3):
        for e in (0, 15, 16, N - 1):
            re = math.fsum(np.concatenate([(V[:, e].real * coef[:, j].real), -(V[:, e].imag * coef[:, j].imag)]))
            # the products above are rounded at 2^-53 of themselves, each at most 1
            assert abs(got[j, e].real - re) <= (4 * 2.0 ** -57 + 2 * 2.0 ** -53) * rows * 2 + 2.0 ** -52 * abs(re)


@pytest.mark.parametrize("n", [96, 163840])       # chunks of 64 entries, and of the largest size, 512
@pytest.mark.parametrize("sign", [1.0, -1.0])
def test_inner_products_of_one_sign(n, sign):
    """A warp's sum of a chunk reaches 2^66 in the integers' unit.  Bar: as above, per entry."""
    need_gpu()
    rng = np.random.default_rng(n)
    V = rng.uniform(0.9, 0.999, (5, n)) + 1j * rng.uniform(0.9, 0.999, (5, n))
    X = sign * (rng.uniform(0.9, 0.999, (3, n)) + 1j * rng.uniform(0.9, 0.999, (3, n)))
    got = _proj(V, _exponents(V), X)
    for a in range(5):
        for j in range(3):
            re = math.fsum(np.concatenate([V[a].real * X[j].real, V[a].imag * X[j].imag]))
            assert abs(got[a, j].real - re) <= (4 * 2.0 ** -57 + 2 * 2.0 ** -53) * n * 2 + 2.0 ** -52 * abs(re) * 16


def test_exponents_beyond_the_range_give_nan_where_they_are():
    need_gpu()
    rng = np.random.default_rng(1)
    V = rng.standard_normal((40, N)) + 1j * rng.standard_normal((40, N))
    coef = rng.standard_normal((40, 4)) + 1j * rng.standard_normal((40, 4))
    X = rng.standard_normal((3, N)) + 1j * rng.standard_normal((3, N))
    want = V.T @ coef
    # a coefficient beyond 2^877: its column; an entry of V (or infinity): its block of 16
    c2 = coef.copy()
    c2[3, 1] = 1e290
    got = _gemm(V, _exponents(V), c2)
    assert np.isnan(got[1]).all() and np.abs(got[[0, 2, 3]] - want.T[[0, 2, 3]]).max() <= 1e-13 * np.abs(want).max()
    V2, E2 = V.copy(), _exponents(V)
    V2[5, 20], E2[1] = np.inf, 2047
    got = _gemm(V2, E2, coef)
    assert np.isnan(got[:, 16:32]).all() and np.isfinite(got[:, :16]).all() and np.isfinite(got[:, 32:]).all()
    X2 = X.copy()
    X2[1, 40] = np.nan
    got, ref = _proj(V, _exponents(V), X2), V.conj() @ X.T
    assert np.isnan(got[:, 1]).all() and np.abs(got[:, [0, 2]] - ref[:, [0, 2]]).max() <= 1e-13 * np.abs(ref).max()


@pytest.mark.parametrize("rows,nx", [(1, 1), (7, 2), (33, 3), (64, 4), (65, 5), (300, 9)])
def test_products_over_a_wide_range(rows, nx):
    """Entries 2^-40 .. 1 apart within their blocks; the error is relative to the largest of a block and vector: 2^-55
    times the number of entries (or rows), and the roundings of numpy's own FP64 products as much."""
    need_gpu()
    rng = np.random.default_rng(rows)
    def draw(shape):
        return (rng.standard_normal(shape) + 1j * rng.standard_normal(shape)) * np.ldexp(1.0, rng.integers(-40, 1, shape))
    V, X, coef = draw((rows, N)), draw((nx, N)), draw((rows, nx))
    vmax = np.abs(V).max()
    got, want = _proj(V, _exponents(V), X), V.conj() @ X.T
    assert np.abs(got - want).max() <= 2 * N * 2.0 ** -52 * vmax * np.abs(X).max()
    got, want = _gemm(V, _exponents(V), coef), (V.T @ coef).T
    assert np.abs(got - want).max() <= 2 * rows * 2.0 ** -52 * vmax * np.abs(coef).max()
