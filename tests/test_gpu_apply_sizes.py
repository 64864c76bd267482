"""FP32 applications on both sides of the sizes at which their kernels stop being launched early: a field's result is the
same bits in a call of any size, and the operator's to 1e-6 of the oracle."""
import numpy as np
import pytest

from oracle.wilson import WilsonOperator
from paper_0901_3512_gb300 import seedcg, workloads as W
from tests.gpu_helpers import dev, host, need_gpu, rel

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,n,multi", [((8, 8, 8, 16), 192, 1), ((8, 8, 8, 16), 193, 1), ((16, 16, 16, 32), 12, 0),
                                          ((16, 16, 16, 32), 13, 0), ((16, 16, 16, 12), 5, 1), ((2, 2, 2, 2), 3, 1)])
def test_single_precision_applications(dims, n, multi):
    need_gpu()
    u = W.gauge_field(dims, 0.5, 81)
    op = WilsonOperator(dims, u, 0.2)
    s = seedcg.Solver(dims, u, 0.2)
    x = dev(W.random_spinors(dims, n, 82))
    y, z = torch.empty_like(x), torch.empty_like(x[:1])
    for code, fn in ((seedcg.OP_D, op.D), (seedcg.OP_DDAG, op.Ddag), (seedcg.OP_M, op.M)):
        s.apply(code, x, y, prec=1, multi=multi)
        for k in (0, n - 1):
            assert rel(host(y[k]), fn(host(x[k]))) <= 1e-6
            s.apply(code, x[k:k + 1].contiguous(), z, prec=1, multi=multi)
            assert torch.equal(z[0], y[k])
    s.close()
