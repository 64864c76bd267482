"""The learned guess's kernels at the edges of their tiles: a lattice smaller than one tile of 32
sites, one that ends in a ragged tile, and one whose weight-gradient CTAs add their tensor-core sums up
more than once.  Bars: those of tests/test_gpu_guess.py (bf16 storage, unit roundoff 2^-9)."""
import numpy as np
import pytest

from oracle.guess import GuessNet, init_weights
from paper_0901_3512_gb300 import seedcg, workloads as W
from tests.gpu_helpers import dev, host, need_gpu, rel

pytestmark = pytest.mark.gpu

U_BF16 = 2.0 ** -9


@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (2, 4, 6, 10), (16, 16, 16, 8)])
def test_forward_and_gradient_at_tile_edges(dims):
    need_gpu()
    u = W.gauge_field(dims, 0.5, 31)
    net = GuessNet(dims, u)
    s = seedcg.Solver(dims, u, 0.2)
    Ws = init_weights(32, scale=1.0)
    seedcg.seedcg_guess_set_weights(s.h, Ws)
    B = W.random_spinors(dims, 1, 33)
    X = W.random_spinors(dims, 1, 34)
    X0 = dev(np.zeros_like(B))
    seedcg.seedcg_guess_predict(s.h, dev(B), X0)
    want, _ = net.forward(Ws, B[0])
    assert rel(host(X0)[0], want) <= 8 * U_BF16
    loss, g = seedcg.seedcg_guess_loss_grad(s.h, dev(B), dev(X))
    lref, gref = net.loss_and_grad(Ws, B, X)
    assert abs(loss - lref) <= 16 * U_BF16 * lref
    for layer, got in enumerate(seedcg.split_weights(g)):
        assert rel(got, gref[layer]) <= 32 * U_BF16, layer
    s.close()
