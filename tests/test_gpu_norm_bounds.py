"""Users, items and queries have one FP32 norm bound: a batch that holds the item of
the largest norm needs no bin parameters of its own."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

rkr = pytest.importorskip("paper_2504_13446_gb300")


def _rows(kind, rng, n, d):
    x = rng.standard_normal((n, d))
    if kind == "integers":
        x = rng.integers(-3, 4, (n, d))
    elif kind == "wide":
        x = x * 2.0 ** -rng.integers(0, 60, (n, d))
    elif kind == "tiny":
        x = x * 1e-30
    elif kind == "one":
        x = x * (np.arange(d) == 0)
    return x.astype(np.float32)


def _allocs(call):
    before = rkr.device_allocations()
    call()
    return rkr.device_allocations() - before


@pytest.mark.parametrize("kind,d", [("normal", 1), ("normal", 7), ("normal", 64), ("normal", 101),
                                    ("normal", 200), ("normal", 256), ("integers", 33),
                                    ("wide", 130), ("tiny", 24), ("one", 40)])
def test_the_largest_item_as_a_query(kind, d):
    rng = np.random.default_rng(d)
    for _ in range(6):
        U, P = _rows(kind, rng, 150, d), _rows(kind, rng, 40, d)
        with rkr.Index(U, P, tau=12, omega=2, s=8) as idx:
            small = _allocs(lambda: idx.query_approx(P * np.float32(0.5), 5, 2.0, single=True))
            top = _allocs(lambda: idx.query_approx(P, 5, 2.0, single=True))
            assert top == small
            users, ranks, off, _ = idx.query_exact(P, 5)
        for q, (wu, wr) in enumerate(oracle.exact_query(U, P, P, np.full(40, 5, np.int32))):
            assert np.array_equal(users[off[q]:off[q + 1]], wu), q
            assert np.array_equal(ranks[off[q]:off[q + 1]], wr), q
