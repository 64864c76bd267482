"""The scalar work around the Lanczos passes: x^1, of which an iteration takes half of the entries two
terms further, after odd and even numbers of iterations; and the reductions, whose integer sums hold in
the middle of FP64's range and leave its ends to plain additions.

Bars: FP64 as the Lanczos scalars elsewhere, 1e-10. FP32: each of the m terms carries the
operator's 128 * 2^-24 (1 + 8 kappa)^2. Scaled systems: the arithmetic is the same but for the
rounding of the sums (2^-53 each), which a hundred iterations at cond(M) < 100 leave below 1e-9.
"""
import numpy as np
import pytest

from oracle.seedcg import seed_lanczos
from oracle.wilson import WilsonOperator
from paper_0901_3512_gb300 import seedcg, workloads as W
from tests.gpu_helpers import dev, host, need_gpu, rel

pytestmark = pytest.mark.gpu
KAPPA = 0.19


def _system(dims, nrhs):
    u = W.gauge_field(dims, 0.5, 101)
    op = WilsonOperator(dims, u, KAPPA)
    B = np.stack([op.Ddag(e).reshape(e.shape) for e in W.z2_sources(dims, nrhs, 102)])
    return u, op, B


@pytest.mark.parametrize("precision", ["fp64", "mixed_v32"])
@pytest.mark.parametrize("m", [1, 11, 12])
@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (2, 4, 6, 10), (8, 8, 8, 8), (12, 12, 12, 16)])
def test_first_solution_after_odd_and_even_iterations(dims, m, precision):
    need_gpu()
    u, op, B = _system(dims, 1)
    ref = seed_lanczos(op.M, B.reshape(1, -1), None, 1e-30, m, 5)
    s = seedcg.Solver(dims, u, KAPPA, precision=precision, past_factor=1.0, stop_after_seed=1, m_max=m)
    X = dev(np.zeros_like(B))
    code, info = s.solve(dev(B), X, 1e-30, 0, 5)
    s.close()
    assert info["m"] == m
    bar = 1e-10 if precision == "fp64" else m * 128 * 2.0 ** -24 * (1 + 8 * KAPPA) ** 2
    assert rel(host(X)[0], ref.X[0]) <= bar


@pytest.mark.parametrize("power", [-472, -300, 300, 450])
def test_scaled_systems_take_the_same_path(power):
    need_gpu()
    dims = (4, 4, 4, 6)
    u, op, B = _system(dims, 3)
    got = []
    for p in (0, power):
        s = seedcg.Solver(dims, u, KAPPA, precision="fp64", past_factor=1.0)
        X = dev(np.zeros_like(B))
        code, info = s.solve(dev(np.ldexp(B.real, p) + 1j * np.ldexp(B.imag, p)), X, 1e-4, 0, 10)
        s.close()
        assert code == seedcg.SEEDCG_OK
        x = host(X)
        got.append((info["m"], np.ldexp(x.real, -p) + 1j * np.ldexp(x.imag, -p)))
    assert got[0][0] == got[1][0]
    assert rel(got[1][1], got[0][1]) <= 1e-9
