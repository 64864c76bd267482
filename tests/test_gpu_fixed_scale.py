"""The FP64 operator's hops alone, for hopping parameters and links of any size: next to a point source there is no
diagonal term, so the whole result is the hop, and it has to be accurate relative to the hop.

Bar: a component is a sum of 6 products and the spin projection, each rounded at most at 2^-53 of |kappa| max|U| max|x|,
in the oracle's chain as in the operator's: 64 * 2^-52 of it covers both with room.
"""
import numpy as np
import pytest

from oracle.wilson import WilsonOperator
from paper_0901_3512_gb300 import seedcg, workloads as W
from tests.gpu_helpers import dev, host, need_gpu

pytestmark = pytest.mark.gpu
DIMS = (4, 2, 4, 6)


@pytest.mark.parametrize("kappa,links,field", [
    (0.2, 1.0, 1.0), (0.49, 1.0, 1.0), (1e-3, 1.0, 1.0), (-1e-6, 1.0, 1.0), (1e-12, 1.0, 1.0), (2.0 ** -97, 1.0, 1.0),
    (1e-40, 1.0, 1.0), (40.0, 1.0, 1.0), (1e30, 1.0, 1.0), (1e-6, 2.0 ** 18, 1e-100), (1e120, 1e-121, 1.0),
    (1e160, 1e160, 1e-240), (1e-160, 1e-160, 1e240), (1e300, 1e-300, 1.0), (1e-300, 1e300, 1.0)])
def test_hops_are_accurate_relative_to_themselves(kappa, links, field):
    need_gpu()
    u = W.gauge_field(DIMS, 0.5, 21) * links
    x = np.zeros((2, W.volume(DIMS), 4, 3), dtype=np.complex128)
    x[0, 5], x[1, -1] = field * W.random_spinors(DIMS, 1, 22)[0, :2]
    op = WilsonOperator(DIMS, u, kappa)
    s = seedcg.Solver(DIMS, u, kappa)
    out = dev(np.zeros_like(x))
    for code, fn in ((seedcg.OP_D, op.D), (seedcg.OP_DDAG, op.Ddag)):
        s.apply(code, dev(x), out, prec=0, multi=1)
        got = host(out)
        for k, src in ((0, 5), (1, W.volume(DIMS) - 1)):
            want = fn(x[k])
            away = np.arange(len(want)) != src
            bar = 64 * 2.0 ** -52 * (abs(kappa) * np.abs(x[k]).max()) * np.abs(u).max()   # no factor under- or overflows
            assert np.isfinite(want).all() and np.abs(want[away]).max() > 0
            assert np.abs(got[k] - want)[away].max() <= bar, np.abs(got[k] - want)[away].max() / bar
            assert np.abs(got[k, src] - want[src]).max() <= 64 * 2.0 ** -52 * np.abs(want).max()
    s.close()
