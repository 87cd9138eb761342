"""Mixed precision with deferred updates, an LP handed over to the whole
tableau: several rows at a time, at every remainder of rows and columns, after
a full history or after phase I with an artificial still basic; the same
outputs, bit for bit, as the form that updates the whole tableau throughout."""
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


def _signed(m, n, seed, phase1=False):
    """Signs beyond the first 1024 entries of A only: planned as a packing LP, and many pivots."""
    g = np.random.default_rng(seed)
    A, b, c = g.uniform(-1, 1, (m, n)), g.uniform(-5 if phase1 else 1, 10, m), g.uniform(-1, 1, n)
    A.reshape(-1)[:1024] = np.abs(A.reshape(-1)[:1024])
    return A, b, c


def _long(m, n, seed, phase1=False):
    """The same with its leading rows loose: several hundred pivots."""
    A, b, c = _signed(m, n, seed, phase1)
    b[:1024 // n + 1] = 1000.0
    return A, b, c


def _redundant(m, n, seed):
    """Two equal rows with b < 0: one's artificial is still basic, at 0, after phase I."""
    g = np.random.default_rng(seed)
    A, b, c = g.uniform(0, 1, (m, n)), g.uniform(50, 100, m), g.uniform(0, 1, n)
    A[-1] = A[-2] = -g.uniform(0.5, 1, n)
    b[-1] = b[-2] = -1.0
    return A, b, c


CASES = {
    "rows_and_columns": [_signed(m, n, 3 * m + n) for m, n in
                         ((120, 120), (121, 127), (122, 128), (123, 129), (129, 191), (255, 64), (258, 257))],
    "phase1": [_signed(130, 110, 5, True), _signed(161, 150, 6, True), _signed(270, 255, 7, True)],
    "long": [_long(m, n, 3 * m + n) for m, n in
             ((120, 120), (121, 127), (122, 128), (123, 129), (129, 191), (255, 96), (258, 257))],
    "long_phase1": [_long(130, 110, 5, True), _long(161, 150, 6, True), _long(270, 255, 7, True)],
    "driven_out": [_redundant(128, 128, 8), _redundant(131, 97, 9), _redundant(190, 200, 10)],
}


@pytest.mark.parametrize("name", CASES)
def test_handed_over_equals_whole_tableau(name):
    batch = W.pack(name, CASES[name])
    mixed = dict(precision=lpb.LP_PREC_FP32_REFINE)
    s = lpb.BatchSolver(batch, opts=lpb.lpb_default_opts(**mixed))
    try:
        assert sum(g["count"] for g in lpb.lp_batch_groups(s.h) if g["kind"] == 4) == batch.num_lps
    finally:
        s.close()
    got = gpu_solve(batch, opts=lpb.lpb_default_opts(**mixed))
    want = gpu_solve(batch, opts=lpb.lpb_default_opts(**mixed, schedule=lpb.LPB_SCHED_STREAMED))
    for key in ("status", "iters", "obj", "x", "y"):
        np.testing.assert_array_equal(got[key], want[key], err_msg=key)
    if name.startswith("long"):
        assert got["iters"].min() > 96  # every LP past a full history
