"""The recount counts its users only for a caller that asks for statistics."""
import ctypes

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

rkr = pytest.importorskip("paper_2504_13446_gb300")


def test_exact_query_without_statistics():
    w = synth.make_workload("approx", n=8000, m=2500, d=40, nq=24)
    lib = rkr.load()
    kk = np.ascontiguousarray(w.k, np.int32)
    users, ranks = (np.zeros(int(kk.sum()), np.int32) for _ in range(2))
    with rkr.Index(w.U, w.P, tau=48, omega=4, s=30, exact_table=True, floor_rank=16) as idx:
        before = lib.rkr_kernel_launches()
        wu, wr, _, st = idx.query_exact(w.Q, w.k)
        with_stats = lib.rkr_kernel_launches() - before
        assert st.recount_users > 0
        before = lib.rkr_kernel_launches()
        rc = lib.rkr_query_exact(idx._h, w.Q.ctypes.data_as(ctypes.c_void_p), len(kk),
                                 kk.ctypes.data_as(ctypes.c_void_p),
                                 users.ctypes.data_as(ctypes.c_void_p),
                                 ranks.ctypes.data_as(ctypes.c_void_p), None, None)
        without = lib.rkr_kernel_launches() - before
    assert rc == 0
    assert np.array_equal(users, wu) and np.array_equal(ranks, wr)
    assert without < with_stats
