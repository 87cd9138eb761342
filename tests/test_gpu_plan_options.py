"""Options and launch forms reach the LPs that deferred updates would take by
default: a requested thread count, lp_batch_set_group_form and
lp_batch_autotune put them in shared memory where they fit, with the same
results."""
import numpy as np
import pytest

from paper_1802_08557_gb300 import lpbatch as lpb
from paper_1802_08557_gb300 import workloads as W

pytestmark = pytest.mark.gpu

KEYS = ("status", "iters", "obj", "x", "y")
MIXED = dict(precision=lpb.LP_PREC_FP32_REFINE)


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1802_08557_gb300 import build
    build.build()
    lpb.load()


def _positive(m, n, seed):
    g = np.random.default_rng(seed)
    return g.uniform(0, 1, (m, n)), g.uniform(1, 100, m), g.uniform(0, 1, n)


def _tiled(lp, count):
    """`count` LPs that share one A, b and c."""
    one = W.pack("one", [lp])
    z = np.zeros(count, np.int64)
    return W.LPBatch("tiled", np.repeat(one.m, count), np.repeat(one.n, count), z, z, z, one.A, one.b, one.c)


def _uneven():
    sizes = [(130, 90), (100, 120), (160, 70), (95, 140), (140, 140), (120, 110), (200, 60), (64, 210), (180, 80)]
    return W.pack("uneven", [_positive(m, n, i) for i, (m, n) in enumerate(sizes)] + [_positive(20, 20, 50)])


def _solve(batch, **opts):
    s = lpb.BatchSolver(batch, opts=lpb.lpb_default_opts(**opts))
    try:
        s.solve()
        r = s.results()
        assert s.plan_info()["internal_errors"] == 0
        return r, lpb.lp_batch_groups(s.h)
    finally:
        s.close()


@pytest.mark.parametrize("name", ["packing", "signed", "mixed"])
def test_block_threads_reaches_every_lp_that_fits(name):
    if name == "packing":
        batch, opts, kind = _tiled(_positive(60, 60, 1), 3000), {}, 1
    elif name == "signed":
        batch, opts, kind = W.mixed_sign_dense(40, 120, 126, start=2, p_phase1=0.0), {}, 1
    else:
        batch, opts, kind = _uneven(), MIXED, 0
    want, _ = _solve(batch, **opts)
    got, groups = _solve(batch, block_threads=96, **opts)
    assert all((g["kind"], g["threads"]) == (kind, 96) for g in groups), groups
    for k in KEYS:
        np.testing.assert_array_equal(got[k], want[k], err_msg=k)


def _deferred(name):
    """A batch whose only group (or, mixed, whose largest) has deferred updates by default; kinds before and after."""
    if name == "packing":
        return _tiled(_positive(60, 60, 1), 6000), {}, 2, 1
    return _uneven(), MIXED, 4, 0


@pytest.mark.parametrize("name", ["packing", "mixed"])
def test_set_group_form_reaches_deferred_groups_that_fit(name):
    batch, opts, kind, whole = _deferred(name)
    s = lpb.BatchSolver(batch, opts=lpb.lpb_default_opts(**opts))
    try:
        s.solve()
        want = s.results()
        before = s.plan_info()
        groups = lpb.lp_batch_groups(s.h)
        at = [i for i, g in enumerate(groups) if g["kind"] == kind]
        assert at, groups
        for threads, persistent in ((32, False), (64, True), (256, False), (256, True)):
            for i in at:
                lpb.lp_batch_set_group_form(s.h, i, threads, persistent)
            now = lpb.lp_batch_groups(s.h)
            assert len(now) == len(groups)
            for i in at:
                assert (now[i]["kind"], now[i]["threads"], now[i]["persistent"]) == (whole, threads, int(persistent))
            s.solve()
            got = s.results()
            for k in KEYS:
                np.testing.assert_array_equal(got[k], want[k], err_msg=k)
            lpb.lp_batch_solve_graph(s.h)
            np.testing.assert_array_equal(s.results()["obj"], want["obj"])
        plan = s.plan_info()
        moved = sum(groups[i]["count"] for i in at)
        assert plan["num_streamed"] == before["num_streamed"] - moved
        assert plan["num_resident"] == before["num_resident"] + moved
    finally:
        s.close()


@pytest.mark.parametrize("name", ["packing", "mixed"])
def test_autotune_covers_deferred_groups_that_fit(name):
    batch, opts, _, _ = _deferred(name)
    s = lpb.BatchSolver(batch, opts=lpb.lpb_default_opts(**opts))
    try:
        s.solve()
        want = s.results()
        lpb.lp_batch_autotune(s.h, rounds=1)
        assert all(g["tuned_ms"] >= 0.0 for g in lpb.lp_batch_groups(s.h))
        s.solve()
        got = s.results()
        for k in KEYS:
            np.testing.assert_array_equal(got[k], want[k], err_msg=k)
    finally:
        s.close()


def test_groups_in_the_workspace_stay_fixed():
    big = W.pack("big", [_positive(300, 250, i) for i in range(3)])
    small = _tiled(_positive(60, 60, 1), 6000)
    for batch, opts in ((big, {}), (big, MIXED), (small, dict(schedule=lpb.LPB_SCHED_STREAMED))):
        s = lpb.BatchSolver(batch, opts=lpb.lpb_default_opts(**opts))
        try:
            for i in range(len(lpb.lp_batch_groups(s.h))):
                with pytest.raises(lpb.LPBError):
                    lpb.lp_batch_set_group_form(s.h, i, 64, False)
        finally:
            s.close()
