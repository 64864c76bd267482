"""Fields go side by side in the rows of a grid, of which there are at most 65535: the last fields of a larger call are
the bits of a call of their own."""
import pytest

from paper_0901_3512_gb300 import seedcg, workloads as W
from tests.gpu_helpers import need_gpu

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
DIMS, VOL = (2, 2, 2, 2), 16


def _fields(n, v, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.view_as_complex(torch.randn(n, v, 4, 3, 2, dtype=torch.float64, device="cuda", generator=g))


def test_reconstruction_of_more_fields_than_grid_rows():
    need_gpu()
    s = seedcg.Solver(DIMS, W.gauge_field(DIMS, 0.5, 67), 0.2)
    n = 65535 + 2
    xo, eta = _fields(n, VOL // 2, 1), _fields(n, VOL, 2)
    full, alone = torch.zeros_like(eta), torch.zeros_like(eta[:2])
    seedcg.seedcg_eo_reconstruct(s.h, xo, eta, full)
    seedcg.seedcg_eo_reconstruct(s.h, xo[-2:].contiguous(), eta[-2:].contiguous(), alone)
    assert torch.equal(full[-2:], alone) and bool((full != 0).all())
    s.close()


@pytest.mark.parametrize("prec", [0, 1])
def test_even_odd_operator_on_more_fields_than_grid_rows(prec):
    need_gpu()
    s = seedcg.Solver(DIMS, W.gauge_field(DIMS, 0.5, 67), 0.2)
    n = 12 * 65535 + 5      # twelve fields per block
    x = _fields(n, VOL // 2, 3)
    out, alone = torch.zeros_like(x), torch.zeros_like(x[:5])
    seedcg.seedcg_apply_eo(s.h, seedcg.EO_MEO, prec, x, out)
    seedcg.seedcg_apply_eo(s.h, seedcg.EO_MEO, prec, x[-5:].contiguous(), alone)
    assert torch.equal(out[-5:], alone) and bool((out != 0).all())
    s.close()
