"""FP64 simplex with deferred updates: every way an element can be formed
(pending pivots in shared memory, in the workspace, after a flush, vectors
outside shared memory), against the oracle bit for bit."""
import numpy as np
import pytest

from paper_1802_08557_gb300 import lpbatch as lpb
from paper_1802_08557_gb300 import workloads as W
from parity_util import compare, gpu_solve, oracle_solve

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1802_08557_gb300 import build
    build.build()
    lpb.load()


def _dense(m, n, seed, signed):
    g = np.random.default_rng(seed)
    if signed:
        return g.uniform(-1, 1, (m, n)), g.uniform(-5, 10, m), g.uniform(-1, 1, n)
    return g.uniform(0, 1, (m, n)), g.uniform(1, 100, m), g.uniform(0, 1, n)


CASES = {
    # one row or column; one element past a warp and past a CTA's threads
    "edges": [(m, n, s) for s in (0, 1) for m, n in ((1, 1), (1, 40), (40, 1), (33, 31), (32, 33), (65, 63), (64, 130))],
    # more pivots than fit before a flush, several flushes, phase I with retired columns
    "flushes": [(60, 60, 1), (75, 40, 1), (40, 75, 1), (120, 118, 1)],
    # pending pivots beyond shared memory (the larger classes)
    "long_history": [(450, 480, 0), (230, 200, 1), (500, 60, 0)],
    # vectors that exceed one CTA's shared memory
    "vectors_in_workspace": [(40, 9000, 0), (12, 9500, 1)],
}


@pytest.mark.parametrize("name", CASES)
def test_deferred_updates_match_the_oracle(name):
    batch = W.pack(name, [_dense(m, n, 7 * i + 1, s) for i, (m, n, s) in enumerate(CASES[name])])
    got = gpu_solve(batch, opts=lpb.lpb_default_opts(schedule=lpb.LPB_SCHED_STREAMED))
    assert got["plan"]["num_streamed"] == batch.num_lps and got["plan"]["internal_errors"] == 0
    assert compare(batch, got, oracle_solve(batch)) == (batch.num_lps, batch.num_lps)
