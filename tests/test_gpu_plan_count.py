"""LPs that fit in shared memory get deferred updates only where a batch has
enough of them: few LPs of one size stay in shared memory, one LP of another
size does not change that, many LPs or many sizes do."""
import numpy as np
import pytest

from paper_1802_08557_gb300 import lpbatch as lpb
from paper_1802_08557_gb300 import workloads as W

pytestmark = pytest.mark.gpu

FP64, MIXED = lpb.LP_PREC_FP64, lpb.LP_PREC_FP32_REFINE


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1802_08557_gb300 import build
    build.build()
    lpb.load()


def _batch(sizes_counts):
    g = np.random.default_rng(5)
    lps = [(g.uniform(0, 1, (m, n)), g.uniform(1, 100, m), g.uniform(0, 1, n)) for m, n, _ in sizes_counts]
    p = W.pack("sizes", lps)
    rep = lambda v: np.repeat(v, [c for _, _, c in sizes_counts])
    return W.LPBatch("repeated", rep(p.m), rep(p.n), rep(p.a_off), rep(p.b_off), rep(p.c_off), p.A, p.b, p.c)


def _deferred(sizes_counts, precision):
    """LPs in a workspace, of all."""
    batch = _batch(sizes_counts)
    s = lpb.BatchSolver(batch, opts=lpb.lpb_default_opts(precision=precision))
    try:
        plan = s.plan_info()
        s.solve()
        r = s.results()
        assert s.plan_info()["internal_errors"] == 0 and (r["status"] == 0).all()
        at = 0
        for _, _, count in sizes_counts:  # copies of one LP: one result
            assert (r["obj"][at:at + count] == r["obj"][at]).all()
            at += count
    finally:
        s.close()
    return plan["num_streamed"]


@pytest.mark.parametrize("precision", [FP64, MIXED])
def test_few_lps_of_one_size_stay_in_shared_memory(precision):
    for size in ((120, 118), (150, 140)):
        assert _deferred([(*size, 200)], precision) == 0
        assert _deferred([(*size, 200), (5, 5, 1)], precision) == 0
    assert _deferred([(120, 118, 60), (140, 130, 60), (110, 120, 60)], precision) == 0


@pytest.mark.parametrize("precision", [FP64, MIXED])
def test_many_lps_or_many_sizes_are_deferred(precision):
    assert _deferred([(150, 140, 2000)], precision) == 2000
    assert _deferred([(150, 140, 2000), (5, 5, 1)], precision) == 2000
    many = [(100 + 9 * i, 130 + 7 * (i % 3), 2) for i in range(12)]
    assert _deferred(many, precision) == 24


def test_large_mixed_lps_need_the_number_too():
    # beyond shared memory in either form: the whole tableau in a workspace slot, or deferred updates
    for count, deferred in ((100, False), (400, True)):
        s = lpb.BatchSolver(_batch([(300, 290, count), (5, 5, 1)]), opts=lpb.lpb_default_opts(precision=MIXED))
        try:
            kinds = {(g["kind"], g["smem_bytes"] > 0) for g in lpb.lp_batch_groups(s.h) if g["count"] == count}
            assert kinds == {(4, deferred)}
        finally:
            s.close()
