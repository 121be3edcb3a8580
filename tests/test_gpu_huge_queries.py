"""Queries whose products with a user exceed the range of float: FP32 scores and
compensated products are then infinite or NaN, the canonical FP64 score is not."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

rkr = pytest.importorskip("paper_2504_13446_gb300")


def test_count_grid_leaves_out_scores_beyond_float():
    # Half of the users lie in the first two coordinates, where the queries are huge
    # and of opposite signs (FP32: inf - inf) and every item is alike, so that their
    # tail lists overflow and they stay open to the recount with no finite interval
    # of u.q.  The other users see ordinary queries.
    n, m, d, nq = 6000, 1500, 24, 64
    rng = np.random.default_rng(8)
    U = synth.workloads.gaussian_rows(rng, n, d, 0.7)
    U[:, :2] = 0
    U[::2] = 0
    U[::2, :2] = np.float32(30)
    P = synth.workloads.gaussian_rows(rng, m, d, 0.7)
    P[:, :2] = np.float32(0.01)
    Q = (synth.workloads.gaussian_rows(rng, nq, d, 0.5) * np.float32(0.2)).astype(np.float32)
    Q[:, 0] = np.float32(1e38)
    Q[:, 1] = -Q[:, 0]
    step = np.where(np.arange(nq) % 2 == 0, np.float32(2e38), np.float32(0))
    Q[:, 1] = np.nextafter(Q[:, 1], -step).astype(np.float32)
    k = rng.integers(1, 40, nq).astype(np.int32)
    with rkr.Index(U, P, tau=32, omega=4, s=20, floor_rank=max(2, m // 32)) as idx:
        rkr.rkr_profile_start()
        try:
            users, ranks, off, _ = idx.query_exact(Q, k)
        finally:
            report = rkr.rkr_profile_stop()
    assert "k_screen<EpiDeep>" in report, "the count grid was not built"
    for q, (wu, wr) in enumerate(oracle.exact_query(U, P, Q, k)):
        assert np.array_equal(users[off[q]:off[q + 1]], wu), q
        assert np.array_equal(ranks[off[q]:off[q + 1]], wr), q


@pytest.mark.parametrize("d,bulk", [(24, 0), (24, 1), (37, 0)])
def test_one_at_a_time_scores_beyond_float(d, bulk):
    rng = np.random.default_rng(d)
    n, m, nq, tau, omega, s = 3000, 700, 6, 40, 3, 20
    U = synth.workloads.gaussian_rows(rng, n, d, 0.7)
    U *= np.float32(30)
    P = synth.workloads.gaussian_rows(rng, m, d, 0.7)
    Q = synth.workloads.gaussian_rows(rng, nq, d, 0.5)
    Q = (Q / np.linalg.norm(Q, axis=1, keepdims=True) * 2e38).astype(np.float32)
    Q[0] = P[5]
    k = np.array([5, 1, 60, 700, 33, 2500], np.int32)
    pos = synth.sample_positions(1, oracle.bucket_sizes(m, omega), s)
    ora = oracle.build_index(U, P, tau, omega, s, pos, fbounds="exact")
    was = rkr.rkr_tuning_get()
    try:
        rkr.rkr_tuning_set(**{**was, "latency_bulk": bulk})
        with rkr.Index(U, P, tau=tau, omega=omega, s=s, sample_pos=pos,
                       exact_table=False) as idx:
            got = idx.query_approx(Q, k, 2.0, single=True)
    finally:
        rkr.rkr_tuning_set(**was)
    off = got["offsets"]
    for q, w in enumerate(oracle.approx_query(ora, U, Q, k, 2.0)):
        sl = slice(off[q], off[q + 1])
        assert got["case"][q] == w["case"] and got["nc"][q] == w["nc"], q
        for a in ("users", "n_low", "n_up", "est"):
            assert np.array_equal(got[a][sl], w[a]), (q, a)


@pytest.mark.parametrize("d,scale_p,exact_table", [
    (24, 1.0, 1), (37, 1.0, 2), (200, 1.0, 2),
    (24, 1e-37, 1),      # grids whose steps lie outside the range of float, too
])
def test_batches_with_scores_beyond_float(d, scale_p, exact_table):
    rng = np.random.default_rng(d)
    n, m, nq, tau, omega, s = 3000, 700, 30, 40, 3, 20
    U = synth.workloads.gaussian_rows(rng, n, d, 0.7) * np.float32(30)
    P = synth.workloads.gaussian_rows(rng, m, d, 0.7) * np.float32(scale_p)
    Q = synth.workloads.gaussian_rows(rng, nq, d, 0.5)
    Q = (Q / np.linalg.norm(Q, axis=1, keepdims=True) * 2e38).astype(np.float32)
    Q[::9] = P[:len(Q[::9])]
    k = rng.integers(1, 400, nq).astype(np.int32)
    k[1] = 2500                                        # past the users with u.q > 0
    pos = synth.sample_positions(1, oracle.bucket_sizes(m, omega), s)
    ora = oracle.build_index(U, P, tau, omega, s, pos, fbounds="exact")
    with rkr.Index(U, P, tau=tau, omega=omega, s=s, sample_pos=pos, exact_table=exact_table,
                   floor_rank=40) as idx:
        got = idx.query_approx(Q, k, 2.0)
        users, ranks, off, _ = idx.query_exact(Q, k)
        pu = rng.integers(0, n, 4000).astype(np.int32)
        pq = rng.integers(0, nq, 4000).astype(np.int32)
        pairs = idx.rank_pairs(Q, pu, pq)
    for q, w in enumerate(oracle.approx_query(ora, U, Q, k, 2.0)):
        sl = slice(off[q], off[q + 1])
        for a in ("users", "n_low", "n_up", "est"):
            assert np.array_equal(got[a][sl], w[a]), (q, a)
    for q, (wu, wr) in enumerate(oracle.exact_query(U, P, Q, k)):
        assert np.array_equal(users[off[q]:off[q + 1]], wu), q
        assert np.array_equal(ranks[off[q]:off[q + 1]], wr), q
    assert np.array_equal(pairs, oracle.ranks(U, P, Q)[pu, pq])
