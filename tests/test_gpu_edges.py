"""Edges of the selection, scan, staging and table kernels, bit for bit against the
FP64 oracle.

Selection: numbers of tied candidates and k around the sort's short form (64), its
bitonic form and the radix search before them, with fewer and with more queries than
SMs.  Scan and staging: dimensions around the vector widths, rows of extreme size.
Tables: widths around the warp's suffix sums.  Saved files: rows padded on the device
are unpadded on disk."""
import os

import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


def _rows(rng, n, d, sigma=0.5):
    g = rng.standard_normal((n, d))
    g /= np.linalg.norm(g, axis=1, keepdims=True)
    return (g * np.exp(sigma * rng.standard_normal((n, 1)))).astype(np.float32)


def _pair(U, P, tau, omega, s, **kw):
    import paper_2504_13446_gb300 as rkr
    pos = synth.sample_positions(1, oracle.bucket_sizes(P.shape[0], omega), s)
    ora = oracle.build_index(U, P, tau, omega, s, pos, fbounds="exact")
    return ora, rkr.Index(U, P, tau=tau, omega=omega, s=s, sample_pos=pos, **kw)


def _check_approx(ora, gpu, U, Q, k, c, single):
    got = gpu.query_approx(Q, k, c, single=single)
    off = got["offsets"]
    for q, w in enumerate(oracle.approx_query(ora, U, Q, k, c)):
        sl = slice(off[q], off[q + 1])
        assert got["case"][q] == w["case"] and got["nc"][q] == w["nc"], q
        for a in ("users", "n_low", "n_up", "est"):
            assert np.array_equal(got[a][sl], w[a]), (q, a)


def _check_exact(gpu, U, P, Q, k):
    users, ranks, off, _ = gpu.query_exact(Q, k)
    for q, (wu, wr) in enumerate(oracle.exact_query(U, P, Q, k)):
        assert np.array_equal(users[off[q]:off[q + 1]], wu), q
        assert np.array_equal(ranks[off[q]:off[q + 1]], wr), q


@pytest.mark.parametrize("c", [1.0, 2.0])
@pytest.mark.parametrize("distinct,n,nq", [(3, 900, 4), (40, 6000, 4), (40, 3000, 160),
                                           (2500, 2500, 6)])
def test_selection_sizes(distinct, n, nq, c):
    rng = np.random.default_rng(distinct + nq)
    d = 19
    U = _rows(rng, distinct, d)[rng.integers(0, distinct, n)]      # users that tie
    P = _rows(rng, 300, d)
    Q = np.concatenate([P[:nq // 2], _rows(rng, nq - nq // 2, d)])
    k = np.array([1, 63, 64, 65, 128, 129, 256, 257, 512, 513, 800, 2])[
        rng.permutation(np.arange(nq) % 12)].astype(np.int32)
    ora, gpu = _pair(U, P, 24, 3, 15, exact_table=True)
    with gpu:
        _check_approx(ora, gpu, U, Q, k, c, single=False)
        _check_exact(gpu, U, P, Q, k)
        if nq < 10:
            _check_approx(ora, gpu, U, Q, k, c, single=True)


def test_selection_beyond_the_survivor_buffer():
    # more than 4,096 survivors of step 3, and k at its largest
    rng = np.random.default_rng(5)
    U, P = _rows(rng, 9000, 12, 0.2), _rows(rng, 400, 12)
    Q = _rows(rng, 3, 12, 0.1)
    k = np.array([4096, 700, 20], np.int32)
    ora, gpu = _pair(U, P, 5, 2, 4, exact_table=True)
    with gpu:
        for c in (1.0, 1.3, 3.0):
            _check_approx(ora, gpu, U, Q, k, c, single=False)
            _check_approx(ora, gpu, U, Q, k, c, single=True)
        _check_exact(gpu, U, P, Q, k)


@pytest.mark.parametrize("d,scale_u,scale_p", [
    (1, 1.0, 1.0), (31, 1.0, 1.0), (33, 1e-18, 1e15), (36, 1e15, 1e-18), (255, 1.0, 1.0),
    (256, 1e-30, 1.0), (4, 1e-40, 1.0),          # the last: subnormal users
])
def test_dimensions_and_magnitudes(d, scale_u, scale_p):
    rng = np.random.default_rng(d)
    U = (_rows(rng, 700, d) * scale_u).astype(np.float32)
    P = (_rows(rng, 260, d) * scale_p).astype(np.float32)
    U[5] = 0
    P[7] = 0
    U[11] *= np.float32(1e-3)
    Q = np.concatenate([P[[3, 7]], (_rows(rng, 3, d) * scale_p).astype(np.float32)])
    k = np.array([1, 20, 7, 64, 33], np.int32)
    ora, gpu = _pair(U, P, 33, 4, 12, exact_table=True)
    with gpu:
        assert np.array_equal(gpu.export("table"), ora["N"])
        _check_approx(ora, gpu, U, Q, k, 2.0, single=False)
        _check_approx(ora, gpu, U, Q, k, 2.0, single=True)
        _check_exact(gpu, U, P, Q, k)


@pytest.mark.parametrize("tau", [2, 31, 32, 33, 64, 257, 1000])
def test_table_widths(tau):
    rng = np.random.default_rng(tau)
    U, P = _rows(rng, 300, 21), _rows(rng, 500, 21)
    Q = np.concatenate([P[:3], _rows(rng, 2, 21)])
    k = np.full(5, 9, np.int32)
    ora, gpu = _pair(U, P, tau, 3, 40)
    with gpu:
        assert np.array_equal(gpu.export("table"), ora["N"])
        _check_approx(ora, gpu, U, Q, k, 1.5, single=False)


@pytest.mark.parametrize("d", [9, 32, 40, 200])
def test_saved_rows_are_unpadded(tmp_path, d):
    import paper_2504_13446_gb300 as rkr
    rng = np.random.default_rng(d)
    n, m = 513, 300
    U, P = _rows(rng, n, d), _rows(rng, m, d)
    Q = np.concatenate([P[:4], _rows(rng, 4, d)])
    k = np.full(8, 11, np.int32)
    a, b = str(tmp_path / "a"), str(tmp_path / "b")
    with rkr.Index(U, P, tau=20, omega=3, s=10, exact_table=True) as idx:
        idx.save(a)
        want = idx.query_exact(Q, k)[:2]
    with rkr.Index.load(a) as idx:
        got = idx.query_exact(Q, k)[:2]
        idx.save(b)
    assert all(np.array_equal(x, y) for x, y in zip(got, want))
    assert open(a, "rb").read() == open(b, "rb").read()


def test_saved_operands_grow_with_their_columns(tmp_path):
    # 16 and 48 operand columns lie at the same pitch on the device; on disk a user's
    # row of 9 or 40 floats and its operands take their own widths
    import paper_2504_13446_gb300 as rkr
    rng = np.random.default_rng(2)
    per_user = []
    for d in (9, 40):
        size = []
        for n in (256, 512):
            path = str(tmp_path / f"{d}_{n}")
            with rkr.Index(_rows(rng, n, d), _rows(rng, 300, d), tau=20, omega=3, s=10,
                           exact_table=False) as idx:
                idx.save(path)
            size.append(os.path.getsize(path))
        per_user.append((size[1] - size[0]) / 256)
    assert per_user[1] - per_user[0] > 4 * (40 - 9)
