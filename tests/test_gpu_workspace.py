"""The workspace of a solve stays within 16 GiB whatever sizes its groups have:
the groups with deferred updates share it."""
import numpy as np
import pytest

from paper_1802_08557_gb300 import lpbatch as lpb
from paper_1802_08557_gb300 import workloads as W

pytestmark = pytest.mark.gpu

CAP = 16 << 30


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1802_08557_gb300 import build
    build.build()
    lpb.load()


def _repeated(sizes_counts, seed):
    """`count` LPs of each size; those of one size share A, b and c."""
    g = np.random.default_rng(seed)
    lps = [(g.uniform(0, 1, (m, m)), g.uniform(1, 100, m), g.uniform(0, 1, m)) for m, _ in sizes_counts]
    p = W.pack("sizes", lps)
    counts = [c for _, c in sizes_counts]
    rep = lambda v: np.repeat(v, counts)
    return W.LPBatch("repeated", rep(p.m), rep(p.n), rep(p.a_off), rep(p.b_off), rep(p.c_off), p.A, p.b, p.c)


# alone, the slots for the larger LPs take the 16 GiB; the smaller ones would like 3 to 5 GB more
@pytest.mark.parametrize("mixed", [False, True])
def test_groups_share_the_workspace(mixed):
    large, small = (5600, 150) if mixed else (4000, 130), (1000, 500)
    batch = _repeated([large, small, (900, 400)], 3)
    opts = lpb.lpb_default_opts(max_iters=3, precision=lpb.LP_PREC_FP32_REFINE if mixed else lpb.LP_PREC_FP64)
    s = lpb.BatchSolver(batch, opts=opts)
    try:
        assert 0 < s.plan_info()["workspace_bytes"] <= (2 if mixed else 1) * CAP  # mixed: and the FP64 re-solve's
        s.solve()
        r = s.results()
        assert s.plan_info()["internal_errors"] == 0
    finally:
        s.close()
    at = 0
    for _, count in (large, small, (900, 400)):
        assert (r["iters"][at:at + count] == 3).all() and (r["obj"][at:at + count] == r["obj"][at]).all()
        at += count
