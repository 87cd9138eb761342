"""The FP64 plan's guess of an LP's sign looks over the whole of A: LPs that
begin with rows of one sign are not taken for packing LPs, others still are,
and the guess changes no result."""
import numpy as np
import pytest

from paper_1802_08557_gb300 import lpbatch as lpb
from paper_1802_08557_gb300 import workloads as W

pytestmark = pytest.mark.gpu

COUNT = 6000


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1802_08557_gb300 import build
    build.build()
    lpb.load()


def _lp(m, n, nonneg_rows, seed):
    g = np.random.default_rng(seed)
    A = g.uniform(-1, 1, (m, n))
    A[:nonneg_rows] = np.abs(A[:nonneg_rows])
    return A, g.uniform(1, 10, m), g.uniform(-1, 1, n)


def _copies(lp):
    """COUNT LPs that share one A, b and c."""
    p = W.pack("one", [lp])
    z = np.zeros(COUNT, np.int64)
    return W.LPBatch("copies", np.repeat(p.m, COUNT), np.repeat(p.n, COUNT), z, z, z, p.A, p.b, p.c)


# signed from the second tenth of the rows on, in the last rows only, and not at all
@pytest.mark.parametrize("m,n,nonneg_rows,kind", [(70, 70, 16, 1), (60, 90, 12, 1), (100, 40, 90, 1), (50, 50, 47, 1),
                                                  (70, 70, 70, 2), (33, 70, 33, 2)])
def test_signs_are_seen_wherever_they_are(m, n, nonneg_rows, kind):
    batch = _copies(_lp(m, n, nonneg_rows, m * n))
    s = lpb.BatchSolver(batch)
    try:
        groups = lpb.lp_batch_groups(s.h)
        assert [g["kind"] for g in groups] == [kind], groups
        s.solve()
        got = s.results()
    finally:
        s.close()
    one = lpb.BatchSolver(batch.subset([0]), opts=lpb.lpb_default_opts(block_threads=64))
    try:
        one.solve()
        want = one.results()
    finally:
        one.close()
    for key, per in (("status", 1), ("iters", 1), ("obj", 1), ("x", n), ("y", m)):
        np.testing.assert_array_equal(got[key].reshape(COUNT, per), np.tile(want[key], (COUNT, 1)), err_msg=key)
