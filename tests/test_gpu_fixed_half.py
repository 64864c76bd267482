"""The FP64 even-odd operator, source and reconstruction at the edges of the fixed point's range (half vectors: neighbours
by half index, hops without a diagonal term, subtracted hops), and the FP32 one on more fields than a block takes.

Bar: a hop is within c = 64 * 2^-52 of kappa max|U| times the largest neighbour component (as on full fields), and what
two or four hops add up to is bounded by k c (1 + 8 kappa max|U|)^hops times the largest component within that many
steps, k = 3 and 6.
"""
import numpy as np
import pytest

from oracle.evenodd import EvenOddOperator
from oracle.wilson import WilsonOperator
from paper_0901_3512_gb300 import seedcg, workloads as W
from tests.gpu_helpers import dev, host, need_gpu, rel

pytestmark = pytest.mark.gpu
C = 64 * 2.0 ** -52


def _near(dims, full, steps):
    """Largest component within `steps` hops of every site; full [n][V][4][3]."""
    m = np.abs(full).max(axis=(2, 3)).reshape((full.shape[0],) + tuple(reversed(dims)))
    for _ in range(steps):
        out = m.copy()
        for ax in range(1, 5):
            out = np.maximum(out, np.maximum(np.roll(m, 1, ax), np.roll(m, -1, ax)))
        m = out
    return m.reshape(full.shape[0], -1)[:, :, None, None]


def _field(dims, n, kind):
    x = W.random_spinors(dims, n, 71)
    rng = np.random.default_rng(72)
    if kind == "spread":
        x *= np.ldexp(1.0, rng.integers(-60, 61, size=(n, x.shape[1], 1, 1)))
        x[:, rng.random(x.shape[1]) < 0.2] = 0.0
    elif kind == "tiny":
        x *= 1e-290
    elif kind == "huge":
        x *= 1e270
    elif kind == "mixed":       # in one tile sites that the fixed point takes and sites that it cannot
        x[:, ::5] *= 1e-290
    return x


def _links(dims, kind):
    u = W.gauge_field(dims, 0.5, 73)
    if kind == "open":
        u[-u.shape[0] // dims[3]:, 3] = 0.0
    elif kind == "unequal":
        u *= np.ldexp(1.0, np.random.default_rng(74).integers(-20, 1, size=u.shape[:2]))[:, :, None, None]
    return u


@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (4, 2, 6, 10), (6, 4, 4, 6)])
@pytest.mark.parametrize("field,links,kappa,n", [
    ("plain", "su3", 0.2, 1), ("spread", "su3", 0.27, 5), ("tiny", "su3", 0.2, 2), ("huge", "su3", 0.2, 2),
    ("mixed", "su3", 0.2, 3), ("plain", "open", 0.2, 13), ("spread", "unequal", 0.2, 2), ("plain", "su3", -1e-3, 2),
    ("plain", "su3", 40.0, 2)])
def test_half_vectors_in_fixed_point(dims, field, links, kappa, n):
    need_gpu()
    u = _links(dims, links)
    eo = EvenOddOperator(WilsonOperator(dims, u, kappa))
    s = seedcg.Solver(dims, u, kappa)
    full = _field(dims, n, field)
    x = np.ascontiguousarray(full[:, eo.odd])
    only_odd = np.stack([eo.embed_odd(v) for v in x])
    scale = 1 + 8 * abs(kappa) * np.abs(u).max()
    out = dev(np.zeros_like(x))
    for code, ref, k, hops in ((seedcg.EO_A, eo.A, 3, 2), (seedcg.EO_ADAG, eo.Adag, 3, 2), (seedcg.EO_MEO, eo.M, 6, 4)):
        seedcg.seedcg_apply_eo(s.h, code, 0, dev(x), out)
        got, want = host(out), np.stack([ref(v) for v in x])
        bar = k * C * scale ** hops * _near(dims, only_odd, hops)[:, eo.odd]
        assert np.all(np.abs(got - want) <= bar), (code, np.max(np.abs(got - want) / np.maximum(bar, 1e-308)))
    seedcg.seedcg_eo_source(s.h, dev(full), out)
    want = np.stack([eo.source(v) for v in full])
    assert np.all(np.abs(host(out) - want) <= C * scale * _near(dims, full, 1)[:, eo.odd])
    back = dev(np.zeros_like(full))
    seedcg.seedcg_eo_reconstruct(s.h, dev(x), dev(full), back)
    want = np.stack([eo.reconstruct(a, b) for a, b in zip(x, full)])
    assert np.all(np.abs(host(back) - want) <= C * scale * _near(dims, full, 1))
    s.close()


def test_non_finite_half_vectors_stay_within_two_hops():
    need_gpu()
    dims = (4, 4, 4, 8)
    u = W.gauge_field(dims, 0.5, 75)
    eo = EvenOddOperator(WilsonOperator(dims, u, 0.2))
    x = np.ascontiguousarray(W.random_spinors(dims, 2, 76)[:, eo.odd])
    clean = np.stack([eo.A(v) for v in x])
    x[0, 17, 1, 2], x[1, 17, 3, 0] = np.nan, np.inf
    s = seedcg.Solver(dims, u, 0.2)
    out = dev(np.zeros_like(x))
    seedcg.seedcg_apply_eo(s.h, seedcg.EO_A, 0, dev(x), out)
    s.close()
    mark = np.zeros((1, W.volume(dims), 1, 1))
    mark[0, eo.odd[17]] = 1.0
    far = _near(dims, mark, 2)[0, eo.odd, 0, 0] == 0
    got = host(out)
    for k in range(2):
        assert not np.isfinite(got[k, 17]).all() and far.any()
        assert np.abs(got[k] - clean[k])[far].max() <= 1e-13 * np.abs(clean[k]).max()


@pytest.mark.parametrize("dims", [(4, 4, 4, 4), (4, 2, 6, 10), (12, 8, 8, 16)])
@pytest.mark.parametrize("n", [3, 12, 13, 25])
def test_fp32_on_more_fields_than_a_block_takes(dims, n):
    """A block takes up to twelve fields, the grid's rows and a loop the others; 1e-5 is the bar of the FP32 operator."""
    need_gpu()
    u = W.gauge_field(dims, 0.5, 77)
    eo = EvenOddOperator(WilsonOperator(dims, u, 0.2))
    s = seedcg.Solver(dims, u, 0.2)
    x = W.random_spinors(dims, n, 78)[:, :W.volume(dims) // 2]
    out = dev(np.zeros_like(x))
    for code, ref in ((seedcg.EO_A, eo.A), (seedcg.EO_MEO, eo.M)):
        seedcg.seedcg_apply_eo(s.h, code, 1, dev(x), out)
        for k in (0, n // 2, n - 1):
            assert rel(host(out)[k], ref(x[k])) <= 1e-5, (code, k)
    s.close()
