"""Hops over links that are weaker than the largest of their field: as accurate as the FP64 chain.

Both are compared with extended precision next to point sources, where the result is the hop alone: the operator's
root-mean-square error, relative to the hops', is at most twice that of the oracle's FP64 chain (which is about 2^-53).
"""
import numpy as np
import pytest

from oracle.wilson import WilsonOperator, gamma
from paper_0901_3512_gb300 import seedcg, workloads as W
from tests.gpu_helpers import dev, host, need_gpu

pytestmark = pytest.mark.gpu
DIMS, KAPPA = (6, 4, 4, 6), 0.2


def _extended(u, x):
    """D x in extended precision (np.clongdouble)."""
    lx, ly, lz, lt = DIMS
    u = u.astype(np.clongdouble).reshape(lt, lz, ly, lx, 4, 3, 3)
    f = x.astype(np.clongdouble).reshape(lt, lz, ly, lx, 4, 3)
    out, one, k = f.copy(), np.eye(4), np.longdouble(KAPPA)
    sign = np.ones(lt)
    for mu in range(4):
        ax = 3 - mu
        fw = np.roll(f, -1, ax)
        bw = np.einsum("tzyxba,tzyxsb->tzyxsa", u[..., mu, :, :].conj(), f)
        bw = np.roll(bw, 1, ax)
        if mu == 3:
            fw[lt - 1] *= -1
            bw[0] *= -1
        fw = np.einsum("tzyxab,tzyxsb->tzyxsa", u[..., mu, :, :], fw)
        out -= k * np.einsum("ij,tzyxja->tzyxia", (one - gamma(mu)).astype(np.clongdouble), fw)
        out -= k * np.einsum("ij,tzyxja->tzyxia", (one + gamma(mu)).astype(np.clongdouble), bw)
    return out.reshape(-1, 4, 3)


@pytest.mark.parametrize("weak", [1.0, 0.5, 2.0 ** -2, 2.0 ** -4, 2.0 ** -7])
def test_hops_over_weak_links(weak):
    need_gpu()
    u = W.gauge_field(DIMS, 0.5, 41)
    v = W.volume(DIMS)
    strong = 3 * v // 4          # the last slices keep links of size 1
    u[:strong] *= weak
    op = WilsonOperator(DIMS, u, KAPPA)
    s = seedcg.Solver(DIMS, u, KAPPA)
    src = np.arange(0, v // 2, 7)
    x = np.zeros((len(src), v, 4, 3), dtype=np.complex128)
    x[np.arange(len(src)), src] = W.random_spinors(DIMS, 1, 42)[0, src]
    out = dev(np.zeros_like(x))
    s.apply(seedcg.OP_D, dev(x), out, prec=0, multi=1)
    s.close()
    e = {"got": 0.0, "chain": 0.0}
    total = 0.0
    for k, at in enumerate(src):
        want = _extended(u, x[k])
        want[at] = 0
        if np.abs(want[strong - v // DIMS[3]:]).max() > 0:
            continue             # a hop across t over a link of size 1
        total += float((np.abs(want) ** 2).sum())
        for name, val in (("got", host(out)[k]), ("chain", op.D(x[k]).reshape(v, 4, 3))):
            d = val - want
            d[at] = 0
            e[name] += float((np.abs(d) ** 2).sum())
    print(weak, np.sqrt(e["got"] / total) * 2.0 ** 53, np.sqrt(e["chain"] / total) * 2.0 ** 53)
    assert 0 < e["got"] <= 4 * e["chain"]
