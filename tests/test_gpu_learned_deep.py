"""The learned cut without the fallback, on queries far below the tail lists.

Every user is then a candidate that needs a recount, none carries a screened score,
and the cut takes t = u.q / ||u|| from FP32 products of the rows.  The test forms
those products, the table's predictions and the cut as the library documents them,
and compares the answer with the exact ranks of the users that are left."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

rkr = pytest.importorskip("paper_2504_13446_gb300")


def _fma(a, b, c):
    # products of floats are exact in long double, and the sum is all but exact
    return (a.astype(np.longdouble) * b + c).astype(np.float32)


def _t(U, q):
    s = np.zeros(len(U), np.float32)
    nn = np.zeros(len(U), np.float32)
    for k in range(U.shape[1]):
        s = _fma(U[:, k], q[k], s)
        nn = _fma(U[:, k], U[:, k], nn)
    return s / np.sqrt(nn)


def _predict(t, tab, grid):
    G = tab.shape[1]
    x = np.clip((t - grid[:, 0]) / grid[:, 1], np.float32(0), np.float32(G - 1))
    j = np.minimum(x.astype(np.int32), G - 2)
    i = np.arange(len(t))
    return _fma(x - j.astype(np.float32), tab[i, j + 1] - tab[i, j], tab[i, j])


def test_cut_takes_t_from_the_rows():
    # one coordinate carries nearly all of every user and query, so the users' t lie
    # within 1e-3 of each other, a few hundred times the error of a screened score
    n, m, d, nq, G, keep = 20000, 1500, 24, 16, 512, 150
    rng = np.random.default_rng(17)
    U = synth.workloads.gaussian_rows(rng, n, d, 0.5)
    U[:, 0] = 30 * np.exp(0.2 * rng.standard_normal(n))
    P = rng.standard_normal((m, d)).astype(np.float32) * np.float32(1000)
    Q = rng.standard_normal((nq, d)).astype(np.float32)
    Q[:, 0] = -2000 * np.exp(0.1 * rng.standard_normal(nq))
    R = (rng.standard_normal((64, d)) / np.sqrt(d)).astype(np.float32)
    net = rkr.Pruner(65, 64, seed=3)
    with rkr.Index(U, P, tau=32, omega=4, s=20, floor_rank=32) as idx:
        net.invert(idx, R, G)
        tab, grid = net.table(n, G)
        users, ranks, off, st = idx.query_exact_learned(net, R, Q, keep, keep, certify=False)
    assert st.deep_queries == nq
    exact = oracle.ranks(U, P, Q)
    for q in range(nq):
        y = _predict(_t(U, Q[q]), tab, grid)
        left = np.flatnonzero(y <= np.partition(y, keep - 1)[keep - 1]).astype(np.int32)
        wu, wr = oracle.select_exact(exact[left, q], keep, left)
        assert np.array_equal(users[off[q]:off[q + 1]], wu), q
        assert np.array_equal(ranks[off[q]:off[q + 1]], wr), q
