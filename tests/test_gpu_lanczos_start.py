"""The vectors of an FP32 Lanczos run are normalised with one rounding of 1 / ||w||, and the first one, r_0 / ||r_0||, in
FP64 whatever the size of the right-hand side."""
import numpy as np
import pytest

from paper_0901_3512_gb300 import seedcg, workloads as W
from tests.gpu_helpers import dev, need_gpu

pytestmark = pytest.mark.gpu
DIMS = (8, 8, 8, 8)
U = 2.0 ** -24    # half a unit in the last place of FP32, relative


def _run(b, eo, m=40, precision="mixed_v32"):
    s = seedcg.Solver(DIMS, W.gauge_field(DIMS, 0.5, 61), 0.2, precision=precision, past_factor=1.0, stop_after_seed=1,
                      m_max=m)
    x = dev(np.zeros_like(b))
    if eo:
        _, info = seedcg.seedcg_solve_eo(s.h, dev(b), x, 1e-30, 0, 0)
    else:
        _, info = s.solve(dev(b), x, 1e-30, 0, 0)
    basis = np.zeros((m, W.volume(DIMS) // (2 if eo else 1), 4, 3), dtype=np.complex128)
    seedcg.seedcg_get_basis(s.h, 0, m, basis)
    a, _, _, _ = seedcg.seedcg_get_lanczos(s.h, m)
    s.close()
    assert info["m"] == m
    return basis.reshape(m, -1), a


@pytest.mark.parametrize("seed", [62, 63, 64])
def test_first_vector_is_rounded_once(seed):
    need_gpu()
    b = W.random_spinors(DIMS, 1, seed)
    V, _ = _run(b, False, m=1)
    r = b.reshape(-1).astype(np.complex64).astype(np.complex128)
    want = r / np.linalg.norm(r)
    for got, w in ((V[0].real, want.real), (V[0].imag, want.imag)):
        assert np.all(np.abs(got - w) <= U * (1 + 2.0 ** -20) * np.abs(w))   # the norm itself is FP64


@pytest.mark.parametrize("eo", [False, True])
@pytest.mark.parametrize("seed", [65, 66])
def test_later_vectors_have_length_one(seed, eo):
    """One rounding of the inverse length moves ||v_i|| by at most U; the entries' own roundings, independent, by
    U / sqrt(n), and the FP32 partial sums behind beta likewise: U / 4 for both."""
    need_gpu()
    V, _ = _run(W.z2_sources(DIMS, 1, seed), eo)
    norms = np.linalg.norm(V, axis=1)
    assert np.abs(norms - 1).max() <= 1.25 * U, np.abs(norms - 1).max() / U


@pytest.mark.parametrize("precision", ["mixed_v32", "fp64"])
@pytest.mark.parametrize("power", [120, -100])
def test_run_does_not_depend_on_the_scale_of_b(power, precision):
    """b times a power of two whose length is beyond FP32 (2^120 times 313 entries' length) is the same run."""
    need_gpu()
    b = W.z2_sources(DIMS, 1, 67) * (1 + 1j)
    V, a = _run(b, False, m=8, precision=precision)
    V2, a2 = _run(b * 2.0 ** power, False, m=8, precision=precision)
    assert np.array_equal(V, V2) and np.array_equal(a, a2)
