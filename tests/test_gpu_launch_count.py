"""seedcg_kernel_launches counts every launch once.  The first solve on a lattice runs the FP32 CG operator's autotuner,
outside any graph: five shapes, once to warm up and three times timed, of the operator's two kernels (four on the
even-odd system).  A second, identical solve (its sums do not depend on the shape) launches just that much less."""
import pytest

from paper_0901_3512_gb300 import seedcg, workloads as W
from tests.gpu_helpers import need_gpu

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("eo,kernels", [(False, 2), (True, 4)])
def test_tuner_launches_are_counted_once(eo, kernels, monkeypatch):
    need_gpu()
    monkeypatch.delenv("SEEDCG_TUNE_CACHE", raising=False)
    dims = (12, 16, 16, 36)
    s = seedcg.Solver(dims, W.gauge_field(dims, 0.5, 51), 0.1, precision="mixed_v32", seed_mode=3)
    b = torch.from_numpy(W.z2_sources(dims, 3, 52)).cuda()
    counts = []
    for _ in range(2):
        x = torch.zeros_like(b)
        before = seedcg.seedcg_kernel_launches()
        if eo:
            seedcg.seedcg_solve_eo(s.h, b, x, 1e-8, 0, 10)
        else:
            s.solve(b, x, 1e-8, 0, 10)
        counts.append(seedcg.seedcg_kernel_launches() - before)
    s.close()
    assert counts[0] - counts[1] == 5 * (1 + 3) * kernels, counts
