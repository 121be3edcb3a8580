"""Calls that fail on the way (an allocation that finds no memory) return with their
stream idle: the caller's arrays are no longer read or written, and the next call is
unaffected."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

rkr = pytest.importorskip("paper_2504_13446_gb300")
torch = pytest.importorskip("torch")


def _calls(idx, w, Qd):
    rng = np.random.default_rng(1)
    pu = rng.integers(0, w.n, 4000).astype(np.int32)
    pq = rng.integers(0, len(w.Q), 4000).astype(np.int32)
    return {
        "approx": lambda: idx.query_approx(Qd, w.k, 2.0)["users"],
        "single": lambda: idx.query_approx(Qd[:40], w.k[:40], 2.0, single=True)["users"],
        "exact": lambda: idx.query_exact(Qd, w.k)[1],
        "pairs": lambda: idx.rank_pairs(Qd, pu, pq),
        "candidates": lambda: idx.query_approx_candidates(Qd[:40], w.k[:40])["users"],
    }


@pytest.mark.parametrize("name", ["approx", "single", "exact", "pairs", "candidates"])
def test_failed_call_leaves_its_stream_idle(name):
    w = synth.make_workload("approx", n=60000, m=3000, d=64, nq=1500)
    Qd = torch.from_numpy(w.Q).cuda()
    stream = torch.cuda.current_stream()
    with rkr.Index(w.U, w.P, tau=64, omega=4, s=30, exact_table=True, floor_rank=32) as idx:
        call = _calls(idx, w, Qd)[name]
        before = rkr.device_allocations()
        want = call()
        count = rkr.device_allocations() - before
        failed = 0
        try:
            for i in range(count):
                rkr.rkr_set_alloc_fault(i)
                try:
                    call()
                except rkr.RKRError:
                    failed += 1
                    assert stream.query(), f"allocation {i} of {count}: work still queued"
                rkr.rkr_set_alloc_fault(-1)
        finally:
            rkr.rkr_set_alloc_fault(-1)
        assert failed >= count // 3
        assert np.array_equal(np.sort(call()), np.sort(want))
