"""The FP64 operator in fixed point at the edges of its range: fields whose sites differ by
many powers of two, values that only the plain FP64 chain can take, links that are zero, of
unequal size, or scaled, tiles that end ragged, and the grid shapes of one and many fields.

Bar: the fixed point's step is 2^-55 of the largest neighbour component and the oracle's
FP64 chain rounds about 20 times at 2^-53, so the two differ by less than 64 * 2^-52 of
(1 + 8 kappa max|U|) times the largest component among a site and its neighbours.
"""
import numpy as np
import pytest

from oracle.wilson import WilsonOperator
from paper_0901_3512_gb300 import seedcg, workloads as W
from tests.gpu_helpers import dev, host, need_gpu

pytestmark = pytest.mark.gpu

DIMS = [(2, 2, 2, 2), (6, 4, 4, 6), (4, 2, 6, 10)]


def _neighbour_max(dims, x):
    m = np.abs(x).max(axis=(2, 3)).reshape((x.shape[0],) + tuple(reversed(dims)))
    out = m.copy()
    for ax in range(1, 5):
        out = np.maximum(out, np.maximum(np.roll(m, 1, ax), np.roll(m, -1, ax)))
    return out.reshape(x.shape[0], -1)


def _field(dims, n, kind):
    x = W.random_spinors(dims, n, 5)
    rng = np.random.default_rng(6)
    v = x.shape[1]
    if kind == "spread":        # sites 2^-60 .. 2^60 apart, some exactly zero
        x *= np.ldexp(1.0, rng.integers(-60, 61, size=(n, v, 1, 1)))
        x[:, rng.random(v) < 0.2] = 0.0
    elif kind == "within":      # components of one site 2^-80 .. 1 apart
        x *= np.ldexp(1.0, rng.integers(-80, 1, size=x.shape))
    elif kind == "tiny":        # below the fixed point's range
        x *= 1e-290
    elif kind == "huge":
        x *= 1e290
    return x


def _links(dims, kind):
    u = W.gauge_field(dims, 0.5, 7)
    rng = np.random.default_rng(8)
    if kind == "open":          # no hop across t
        u[-u.shape[0] // dims[3]:, 3] = 0.0
    elif kind == "unequal":     # links 2^-20 .. 2^3 in size: beyond the fixed point's range
        u *= np.ldexp(1.0, rng.integers(-20, 4, size=u.shape[:2]))[:, :, None, None]
    elif kind == "scaled":      # not unitary, within its range
        u *= rng.uniform(0.5, 3.0, size=u.shape[:2])[:, :, None, None]
    return u


@pytest.mark.parametrize("dims", DIMS)
@pytest.mark.parametrize("field,links,kappa,n", [
    ("plain", "su3", 0.2, 1), ("spread", "su3", 0.27, 5), ("within", "su3", 0.2, 2), ("tiny", "su3", 0.2, 2),
    ("huge", "su3", 0.2, 2), ("plain", "open", 0.2, 3), ("spread", "unequal", 0.2, 2), ("plain", "scaled", 0.15, 13),
    ("plain", "su3", 0.0, 2), ("plain", "su3", -1e-3, 2), ("plain", "su3", 40.0, 2)])
def test_operator_in_fixed_point(dims, field, links, kappa, n):
    need_gpu()
    u = _links(dims, links)
    x = _field(dims, n, field)
    op = WilsonOperator(dims, u, kappa)
    s = seedcg.Solver(dims, u, kappa)
    out = dev(np.zeros_like(x))
    scale = 1.0 + 8.0 * abs(kappa) * np.abs(u).max()
    bar = 64 * 2.0 ** -52 * scale * _neighbour_max(dims, x)[:, :, None, None]
    for code, fn in ((seedcg.OP_D, op.D), (seedcg.OP_DDAG, op.Ddag)):
        s.apply(code, dev(x), out, prec=0, multi=1)
        got = host(out)
        want = np.stack([fn(v) for v in x])
        assert np.all(np.abs(got - want) <= bar), np.max(np.abs(got - want) / np.maximum(bar, 1e-300))
        single = dev(np.zeros_like(x[:1]))
        s.apply(code, dev(x[:1]), single, prec=0, multi=0)
        assert np.array_equal(host(single)[0], got[0])   # sums are exact: no order, no grid shape matters
    s.close()


def test_non_finite_values_stay_where_the_stencil_puts_them():
    need_gpu()
    dims = (4, 4, 4, 8)
    v = W.volume(dims)
    u = W.gauge_field(dims, 0.5, 9)
    op = WilsonOperator(dims, u, 0.2)
    x = W.random_spinors(dims, 2, 10)
    clean = [op.D(f) for f in x]
    x[0, 37, 1, 2] = np.nan
    x[1, 37, 3, 0] = np.inf
    s = seedcg.Solver(dims, u, 0.2)
    out = dev(np.zeros_like(x))
    s.apply(seedcg.OP_D, dev(x), out, prec=0, multi=1)
    got = host(out)
    mark = np.zeros((1, v, 1, 1))
    mark[0, 37] = 1.0
    touched = _neighbour_max(dims, mark)[0] > 0
    for k in range(2):
        assert not np.isfinite(got[k, 37]).all()
        assert all(not np.isfinite(got[k, y]).all() for y in np.nonzero(touched)[0])
        ok = ~touched
        assert np.abs(got[k][ok] - clean[k].reshape(v, 4, 3)[ok]).max() <= 1e-13 * np.abs(clean[k]).max()
    s.close()


@pytest.mark.parametrize("dims,nrhs,eo", [((2, 2, 2, 2), 3, 0), ((2, 2, 2, 4), 4, 1), ((2, 4, 6, 10), 6, 0),
                                          ((8, 8, 8, 8), 8, 0), ((8, 8, 8, 8), 3, 1)])
def test_fp64_basis_products_in_fixed_point(dims, nrhs, eo):
    """Re-orthogonalisation (V^dag [v, f] and the subtraction) and the seeds V T^-1 V^dag r against
    numpy's FP64 products with the stored basis itself: one block of entries, ragged chunks, one to four
    vectors per pass, rows in one segment and in several.  Bars: V^dag V = 1 to the 1e-10 that step 8
    promises, and seeds to 1e-9, which covers cond(T) below 1e4 times the rounding of either side."""
    need_gpu()
    u = W.gauge_field(dims, 0.5, 81)
    eta = W.point_sources(dims, nrhs) if not eo else W.z2_sources(dims, nrhs, 82)
    s = seedcg.Solver(dims, u, 0.19, precision="fp64", past_factor=1.0, stop_after_seed=1, m_max=400)
    X = dev(np.zeros_like(eta))
    if eo:
        code, info = seedcg.seedcg_solve_eo(s.h, dev(eta), X, 1e-8, 0, 5)
    else:
        B = dev(np.zeros_like(eta))
        s.apply(seedcg.OP_DDAG, dev(eta), B, prec=0, multi=1)
        code, info = s.solve(B, X, 1e-8, 0, 5)
    m, v = info["m"], W.volume(dims) // (2 if eo else 1)
    assert info["po_count"] > 0
    basis = np.zeros((m, v, 4, 3), dtype=np.complex128)
    seedcg.seedcg_get_basis(s.h, 0, m, basis)
    V = basis.reshape(m, -1)
    last = 5 * (m // 5)          # vectors up to the last re-orthogonalisation
    gram = V[:last].conj() @ V[:last].T
    assert np.abs(gram[last - 1] - np.eye(last)[last - 1]).max() <= 1e-10
    if not eo:
        a, b, _, _ = seedcg.seedcg_get_lanczos(s.h, m)
        T = np.diag(a) + np.diag(b[:m - 1], 1) + np.diag(b[:m - 1], -1)
        Bh = host(B).reshape(nrhs, -1)
        want = (V.T @ np.linalg.solve(T, V.conj() @ Bh[1:].T)).T
        got = host(X).reshape(nrhs, -1)[1:]
        for g, w in zip(got, want):
            assert np.linalg.norm(g - w) <= 1e-9 * np.linalg.norm(w)
    s.close()
