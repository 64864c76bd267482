"""The FP64 operator on fields of which one spin is far above the others.  Spin s of D x takes the spins s, s ^ 2 and
s ^ 3 of a site and its neighbours, so with a large spin s ^ 1 alone it is small, and has to be as accurate as the sums
of small numbers that it is.

Bar: 64 * 2^-52 of (1 + 8 kappa max|U|) times the largest of those three spins among a site and its neighbours (the
FP64 chain rounds about 20 times at 2^-53).
"""
import numpy as np
import pytest

from oracle.evenodd import EvenOddOperator
from oracle.wilson import WilsonOperator
from paper_0901_3512_gb300 import seedcg, workloads as W
from tests.gpu_helpers import dev, host, need_gpu

pytestmark = pytest.mark.gpu


def _bar(dims, x, spin, scale):
    m = np.abs(np.delete(x, spin ^ 1, axis=2)).max(axis=(2, 3)).reshape((x.shape[0],) + tuple(reversed(dims)))
    out = m.copy()
    for ax in range(1, 5):
        out = np.maximum(out, np.maximum(np.roll(m, 1, ax), np.roll(m, -1, ax)))
    return 64 * 2.0 ** -52 * scale * out.reshape(x.shape[0], -1)[:, :, None]


@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (4, 2, 6, 10)])
@pytest.mark.parametrize("spin,below", [(0, 30), (1, 23), (2, 45), (3, 70)])
def test_a_small_spin_keeps_its_digits(dims, spin, below):
    need_gpu()
    kappa = 0.2
    u = W.gauge_field(dims, 0.5, 91)
    x = W.random_spinors(dims, 2, 92) * 2.0 ** -below
    x[:, :, spin ^ 1] *= 2.0 ** below
    scale = 1 + 8 * kappa * np.abs(u).max()
    bar = _bar(dims, x, spin, scale)
    op = WilsonOperator(dims, u, kappa)
    eo = EvenOddOperator(op)
    s = seedcg.Solver(dims, u, kappa)
    out = dev(np.zeros_like(x))
    for code, fn in ((seedcg.OP_D, op.D), (seedcg.OP_DDAG, op.Ddag)):
        s.apply(code, dev(x), out, prec=0, multi=1)
        got = host(out).reshape(x.shape)
        want = np.stack([fn(v) for v in x]).reshape(x.shape)
        assert np.all(np.abs(got - want)[:, :, spin] <= bar)
    # half vectors: the source of the even-odd system is one subtracted hop
    phi = dev(np.zeros_like(x[:, eo.odd]))
    seedcg.seedcg_eo_source(s.h, dev(x), phi)
    want = np.stack([eo.source(v) for v in x])
    assert np.all(np.abs(host(phi) - want)[:, :, spin] <= bar[:, eo.odd])
    s.close()
