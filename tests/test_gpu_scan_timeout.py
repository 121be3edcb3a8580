"""A stage wait of the bulk-staged scan that runs out.

rkr_set_wait_limit(0) makes the consumer warps give up before their first stage has
landed.  With at most one chunk of 64 users per SM the producer itself waits for no
free stage; it still waits for the copy it issued, so nothing is in flight when the
CTA ends.  The call reports RKR_ETIMEOUT, and the next calls succeed unchanged."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

rkr = pytest.importorskip("paper_2504_13446_gb300")

ETIMEOUT = 4
KEYS = ("users", "n_low", "n_up", "est", "case", "nc")


@pytest.fixture
def bulk():
    was = rkr.rkr_tuning_get()
    rkr.rkr_tuning_set(**{**was, "latency_bulk": 1})
    try:
        yield
    finally:
        rkr.rkr_set_wait_limit(-1)
        rkr.rkr_tuning_set(**was)


def _index():
    w = synth.make_workload("approx", n=4000, m=900, d=48, nq=5)
    return w, rkr.Index(w.U, w.P, tau=40, omega=3, s=30, exact_table=False)


def test_calls_report_the_timeout_and_recover(bulk):
    w, idx = _index()
    with idx:
        want = idx.query_approx(w.Q, w.k, 2.0, single=True)
        for _ in range(2):
            rkr.rkr_set_wait_limit(0)
            with pytest.raises(rkr.RKRError) as e:
                idx.query_approx(w.Q, w.k, 2.0, single=True)
            assert e.value.status == ETIMEOUT
            with pytest.raises(rkr.RKRError) as e:
                idx.query_approx_candidates(w.Q, w.k)
            assert e.value.status == ETIMEOUT
            rkr.rkr_set_wait_limit(-1)
            got = idx.query_approx(w.Q, w.k, 2.0, single=True)
            for key in KEYS:
                assert (got[key] == want[key]).all(), key


def test_session_survives_a_timeout(bulk):
    # the counts of a replay that timed out carry over to no later one, and neither
    # does its error
    w, idx = _index()
    with idx, rkr.Session(idx, max_k=int(w.k.max())) as sess:
        want = [sess.query(w.Q[q], int(w.k[q])) for q in range(len(w.Q))]
        for _ in range(3):
            rkr.rkr_set_wait_limit(0)
            for q in range(len(w.Q)):
                with pytest.raises(rkr.RKRError) as e:
                    sess.query(w.Q[q], int(w.k[q]))
                assert e.value.status == ETIMEOUT
            rkr.rkr_set_wait_limit(-1)
            for q in range(len(w.Q)):
                got = sess.query(w.Q[q], int(w.k[q]))
                for key in KEYS:
                    assert (got[key] == want[q][key]).all(), (q, key)
