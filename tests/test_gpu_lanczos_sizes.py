"""The Lanczos operator kernels at the sizes where the blocks per SM, and with them the
neighbours in flight, change, and on either side of the iterations that keep v_i apart from
its row of V: the recurrence beta_i v_{i+1} = M v_i - alpha_i v_i - beta_{i-1} v_{i-1} with
the stored basis, M by the oracle in FP64.

Bar, in the 2-norm: D and D^dag are sums of 9 terms of which each takes about 12 rounded
steps, at most 128 * 2^-24 of (1 + 8 kappa)^2 with the update and the re-orthogonalisation;
a basis in BF16 adds 2^-9 of each of the four vectors times its coefficient.
"""
import numpy as np
import pytest

from oracle.wilson import WilsonOperator
from paper_0901_3512_gb300 import seedcg, workloads as W
from tests.gpu_helpers import dev, need_gpu

pytestmark = pytest.mark.gpu
KAPPA = 0.2


@pytest.mark.parametrize("precision", ["mixed_v32", "mixed_vbf16"])
@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (2, 6, 10, 14), (16, 8, 8, 38), (14, 14, 10, 20), (16, 16, 6, 38),
                                  (14, 14, 14, 22)])
def test_lanczos_recurrence_over_the_sizes(dims, precision):
    need_gpu()
    u = W.gauge_field(dims, 0.5, 91)
    b = W.z2_sources(dims, 1, 92)
    s = seedcg.Solver(dims, u, KAPPA, precision=precision, past_factor=1.0, stop_after_seed=1, m_max=12)
    X = dev(np.zeros_like(b))
    code, info = s.solve(dev(b), X, 1e-30, 0, 5)
    m = info["m"]
    assert m == 12 and info["po_count"] == 2
    basis = np.zeros((m,) + b.shape[1:], dtype=np.complex128)
    seedcg.seedcg_get_basis(s.h, 0, m, basis)
    a, be, _, _ = seedcg.seedcg_get_lanczos(s.h, m)
    s.close()
    op = WilsonOperator(dims, u, KAPPA)
    V = basis.reshape(m, -1)
    for i in (0, 3, 4, 5, 9, 10):
        av = op.M(V[i])
        want = av - a[i] * V[i] - (be[i - 1] * V[i - 1] if i else 0)
        bar = 128 * 2.0 ** -24 * (1 + 8 * KAPPA) ** 2
        if precision == "mixed_vbf16":
            bar += 2.0 ** -9 * (np.linalg.norm(av) + a[i] + be[i] + (be[i - 1] if i else 0))
        assert np.linalg.norm(be[i] * V[i + 1] - want) <= bar, (i, bar)
