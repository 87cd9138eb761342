"""Mixed precision with deferred updates (uneven batches of packing LPs): the
same outputs, bit for bit, as the form that updates the whole tableau."""
import numpy as np
import pytest

from paper_1802_08557_gb300 import lpbatch as lpb
from paper_1802_08557_gb300 import workloads as W
from parity_util import gpu_solve

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1802_08557_gb300 import build
    build.build()
    lpb.load()


def _positive(m, n, seed, lo=0.0, hi=1.0):
    g = np.random.default_rng(seed)
    return g.uniform(lo, hi, (m, n)), g.uniform(1, 100, m), g.uniform(lo, hi, n)


def _infeasible(m, n, seed):
    A, b, c = _positive(m, n, seed)
    b[5::31] = -0.5  # A >= 0: no point satisfies these rows (phase I, Farkas certificate)
    return A, b, c


def _unbounded(m, n, seed):
    A, b, c = _positive(m, n, seed)
    A[:, 7] = 0.0  # no row bounds variable 7
    return A, b, c


CASES = {
    # class edges: 128 / 129, 256 / 257 rows or columns, the shortest sides that qualify
    "edges": [(128, 128), (129, 100), (100, 129), (256, 60), (60, 257), (32, 380), (380, 32), (450, 470)],
    # more pivots than are kept pending: handed over to the whole tableau
    # (signed beyond the part of A that the plan looks at), phase I among them
    "handed_over": [],
}


def _signed_later(m, n, seed, phase1):
    g = np.random.default_rng(seed)
    A, b, c = g.uniform(-1, 1, (m, n)), g.uniform(-5 if phase1 else 1, 10, m), g.uniform(-1, 1, n)
    A.reshape(-1)[:1024] = np.abs(A.reshape(-1)[:1024])
    return A, b, c


@pytest.mark.parametrize("name", [*CASES, "halts"])
def test_deferred_equals_whole_tableau(name):
    if name == "halts":
        lps = [_infeasible(140, 150, 3), _unbounded(200, 130, 4), _infeasible(300, 290, 5), _unbounded(130, 400, 6)]
    elif name == "handed_over":
        lps = [_signed_later(120, 120, 1, False), _signed_later(130, 110, 2, True), _signed_later(150, 160, 3, True),
               _signed_later(300, 280, 4, False)]
    else:
        lps = [_positive(*a[:2], 11 * i + 1, *a[2:]) for i, a in enumerate(CASES[name])]
    batch = W.pack(name, lps)
    mixed = dict(precision=lpb.LP_PREC_FP32_REFINE)
    got = gpu_solve(batch, opts=lpb.lpb_default_opts(**mixed))
    s = lpb.BatchSolver(batch, opts=lpb.lpb_default_opts(**mixed))
    try:
        groups = [g for g in lpb.lp_batch_groups(s.h) if g["kind"] == 4]
        assert sum(g["count"] for g in groups) == len(lps) and all(g["smem_bytes"] > 0 for g in groups), groups
    finally:
        s.close()
    want = gpu_solve(batch, opts=lpb.lpb_default_opts(**mixed, schedule=lpb.LPB_SCHED_STREAMED))
    for key in ("status", "iters", "obj", "x", "y"):
        np.testing.assert_array_equal(got[key], want[key], err_msg=key)
    assert got["plan"]["num_fallback"] == want["plan"]["num_fallback"]
    if name == "handed_over":
        assert got["iters"].max() > 48
    if name == "halts":
        assert got["status"].tolist() == [1, 2, 1, 2]
