"""Exact queries with many open candidates per user: the count grid of the recount.

Fresh queries of small norm have u.q near 0 for every user, far below the tail
lists, so nearly every user is a candidate of every query and the library bounds
their counts on a per-user grid first (an EpiDeep screen inside the query)."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


def _grid_used(rkr, call):
    rkr.rkr_profile_start()
    try:
        out = call()
    finally:
        report = rkr.rkr_profile_stop()
    return out, "k_screen<EpiDeep>" in report


@pytest.mark.parametrize("n,m,d,nq,scale", [
    (2049, 1500, 37, 64, 0.3),    # ragged rows, columns and dimension
    (5000, 300, 64, 40, 0.05),    # narrow spread: many open intervals
    (4096, 257, 16, 48, 0.5),     # one item past a column tile
    (6000, 700, 20, 30, 0.0),     # zero queries: every u.q ties at 0
])
def test_exact_with_count_grid(n, m, d, nq, scale):
    import paper_2504_13446_gb300 as rkr
    rng = np.random.default_rng(n + d)
    U = synth.workloads.gaussian_rows(rng, n, d, 0.7)
    P = synth.workloads.gaussian_rows(rng, m, d, 0.7)
    Q = (synth.workloads.gaussian_rows(rng, nq, d, 0.5) * np.float32(scale)).astype(np.float32)
    Q[::7] = P[rng.choice(m, len(Q[::7]))]         # some items among them
    k = rng.integers(1, 40, nq).astype(np.int32)
    with rkr.Index(U, P, tau=32, omega=4, s=20, floor_rank=max(2, m // 32)) as idx:
        (users, ranks, off, st), used = _grid_used(rkr, lambda: idx.query_exact(Q, k))
    assert used, "the count grid was not built"
    for q, (wu, wr) in enumerate(oracle.exact_query(U, P, Q, k)):
        assert np.array_equal(users[off[q]:off[q + 1]], wu)
        assert np.array_equal(ranks[off[q]:off[q + 1]], wr)


def test_count_grid_with_subsets():
    import paper_2504_13446_gb300 as rkr
    n, m, d, nq = 5000, 900, 50, 48
    rng = np.random.default_rng(3)
    U = synth.workloads.gaussian_rows(rng, n, d, 0.7)
    P = synth.workloads.gaussian_rows(rng, m, d, 0.7)
    Q = (synth.workloads.gaussian_rows(rng, nq, d, 0.5) * np.float32(0.2)).astype(np.float32)
    k = rng.integers(1, 30, nq).astype(np.int32)
    subsets = [np.sort(rng.choice(n, int(rng.integers(2000, n)), replace=False)).astype(np.int32)
               for _ in range(nq)]
    with rkr.Index(U, P, tau=32, omega=4, s=20, floor_rank=30) as idx:
        (users, ranks, off, _), used = _grid_used(
            rkr, lambda: idx.query_exact(Q, k, subsets=subsets))
    assert used, "the count grid was not built"
    for q in range(nq):
        wu, wr = oracle.exact_query(U[subsets[q]], P, Q[q:q + 1], k[q:q + 1])[0]
        assert np.array_equal(users[off[q]:off[q + 1]], subsets[q][wu])
        assert np.array_equal(ranks[off[q]:off[q + 1]], wr)
