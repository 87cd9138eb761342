"""Which FP64 LPs that fit in shared memory get deferred updates: by sign, shape
and size, the same from host and from device memory; and the results are those
of the shared-memory form bit for bit."""
import numpy as np
import pytest

from paper_1802_08557_gb300 import lpbatch as lpb
from paper_1802_08557_gb300 import workloads as W

pytestmark = pytest.mark.gpu

COUNT = 2000
RESIDENT, DEFERRED = 1, 2


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1802_08557_gb300 import build
    build.build()
    lpb.load()


def _copies(m, n, signed, count):
    """`count` LPs that share one A, b and c."""
    g = np.random.default_rng(m * 10007 + n)
    lo = -1 if signed else 0
    p = W.pack("one", [(g.uniform(lo, 1, (m, n)), g.uniform(1, 10, m), g.uniform(lo, 1, n))])
    z = np.zeros(count, np.int64)
    return W.LPBatch("copies", np.repeat(p.m, count), np.repeat(p.n, count), z, z, z, p.A, p.b, p.c)


CASES = [
    # signed: square, tall and short-rowed LPs stay in shared memory, wide ones and d <= 128 do not
    (True, 130, 130, RESIDENT), (True, 128, 127, DEFERRED), (True, 112, 127, DEFERRED), (True, 700, 32, RESIDENT),
    (True, 225, 64, RESIDENT), (True, 250, 90, RESIDENT), (True, 110, 160, RESIDENT), (True, 64, 225, DEFERRED),
    (True, 24, 1000, DEFERRED), (True, 16, 1400, RESIDENT), (True, 1100, 12, RESIDENT), (True, 1450, 10, DEFERRED),
    # packing LPs: all but rows beyond 1024 entries
    (False, 130, 130, DEFERRED), (False, 700, 32, DEFERRED), (False, 16, 900, DEFERRED), (False, 24, 600, DEFERRED),
    (False, 8, 1600, RESIDENT), (False, 20, 1100, RESIDENT), (False, 1600, 8, DEFERRED), (False, 750, 20, DEFERRED),
]


@pytest.mark.parametrize("device", [True, False])
def test_rule(device):
    for signed, m, n, kind in CASES:
        s = lpb.BatchSolver(_copies(m, n, signed, COUNT), device_data=device)
        try:
            groups = lpb.lp_batch_groups(s.h)
            assert [g["kind"] for g in groups] == [kind], (signed, m, n, groups)
        finally:
            s.close()


@pytest.mark.parametrize("signed,m,n", [(c[0], c[1], c[2]) for c in CASES if c[3] == DEFERRED])
def test_deferred_equals_resident(signed, m, n):
    got = []
    for opts, count in (({}, COUNT), (dict(block_threads=128), 1)):
        s = lpb.BatchSolver(_copies(m, n, signed, count), opts=lpb.lpb_default_opts(**opts))
        try:
            s.solve()
            got.append(s.results())
            assert s.plan_info()["internal_errors"] == 0
        finally:
            s.close()
    for key, per in (("status", 1), ("iters", 1), ("obj", 1), ("x", n), ("y", m)):
        np.testing.assert_array_equal(got[0][key].reshape(COUNT, per), np.tile(got[1][key], (COUNT, 1)), err_msg=key)
