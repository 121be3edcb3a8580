"""Batches whose candidates take several chunks: every chunk's screen reads its own
queries' operands, in either form (split_cat), without the skim list (skip level 30),
as deep queries (the default level) and as listed ones."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

rkr = pytest.importorskip("paper_2504_13446_gb300")


@pytest.mark.parametrize("d,split_cat,level", [(72, 1, 30), (72, 0, 30), (200, 1, 30),
                                               (72, 1, 0), (72, 1, 7)])
def test_batches_in_several_chunks(d, split_cat, level):
    rng = np.random.default_rng(d)
    n, m, nq, tau, omega, s = 12000, 900, 330, 40, 3, 20
    U = synth.workloads.gaussian_rows(rng, n, d, 0.5)
    P = synth.workloads.gaussian_rows(rng, m, d, 0.5)
    Q = P[rng.choice(m, nq, replace=False)]
    k = rng.integers(3500, 4097, nq).astype(np.int32)     # together more than 2^20
    pos = synth.sample_positions(1, oracle.bucket_sizes(m, omega), s)
    ora = oracle.build_index(U, P, tau, omega, s, pos, fbounds="exact")
    was = rkr.rkr_tuning_get()
    try:
        rkr.rkr_tuning_set(**{**was, "skip_level": level, "cand_budget_log2": 20,
                              "split_cat": split_cat})
        with rkr.Index(U, P, tau=tau, omega=omega, s=s, sample_pos=pos, floor_rank=60) as idx:
            got = idx.query_approx(Q, k, 2.0)
            users, ranks, off, _ = idx.query_exact(Q, k)
    finally:
        rkr.rkr_tuning_set(**was)
    exact = oracle.exact_query(U, P, Q, k)
    for q, w in enumerate(oracle.approx_query(ora, U, Q, k, 2.0)):
        sl = slice(off[q], off[q + 1])
        for a in ("users", "n_low", "n_up", "est"):
            assert np.array_equal(got[a][sl], w[a]), (q, a)
        assert np.array_equal(users[sl], exact[q][0]) and np.array_equal(ranks[sl], exact[q][1]), q
