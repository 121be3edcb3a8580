"""The list screen's column tiles, in norm order and from both ends in turn (by the
number of K chunks of a tile), at few, odd and even numbers of tiles."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d", [24, 128, 129, 200])
@pytest.mark.parametrize("m", [200, 256, 257, 700, 1100])
def test_lists_of_either_order(d, m):
    import paper_2504_13446_gb300 as rkr
    rng = np.random.default_rng(d + m)
    U = synth.workloads.gaussian_rows(rng, 300, d, 0.7)
    P = synth.workloads.gaussian_rows(rng, m, d, 0.7)
    Q = np.concatenate([P[rng.choice(m, 6)], synth.workloads.gaussian_rows(rng, 6, d, 0.5)])
    k = rng.integers(1, 60, 12).astype(np.int32)
    with rkr.Index(U, P, tau=32, omega=4, s=20, exact_table=1) as idx:
        xlo, xhi = idx.export("xlo"), idx.export("xhi")
        users, ranks, off, _ = idx.query_exact(Q, k)
        x0, dx = idx.export("xgrid").T
    above = (oracle.scores(U, P)[:, :, None] > (x0[:, None, None] + dx[:, None, None] *
                                                np.arange(xlo.shape[1]))).sum(1)
    assert (xlo <= above).all() and (above <= xhi).all()
    for q, (wu, wr) in enumerate(oracle.exact_query(U, P, Q, k)):
        assert np.array_equal(users[off[q]:off[q + 1]], wu), q
        assert np.array_equal(ranks[off[q]:off[q + 1]], wr), q
