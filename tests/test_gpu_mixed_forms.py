"""The one-warp mixed-precision kernel's two codes, chosen by the majority of a
batch's LPs on one side of a shared-memory line (14 KB): the same outputs, bit
for bit, as the form with the tableau in a global workspace."""
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


# (m, n): a single row or column, 50 x 50 at the line (phase I takes it past), long sides, the largest one-warp LP
@pytest.mark.parametrize("m,n", [(1, 1), (3, 2), (50, 50), (51, 51), (30, 86), (86, 30), (62, 40), (89, 90)])
def test_both_unrollings_match_the_workspace_form(m, n):
    batch = W.mixed_sign_dense(60, m, n, start=17 * m + n, p_phase1=0.4)
    got = gpu_solve(batch, opts=lpb.lpb_default_opts(precision=lpb.LP_PREC_FP32_REFINE))
    want = gpu_solve(batch, opts=lpb.lpb_default_opts(precision=lpb.LP_PREC_FP32_REFINE,
                                                      schedule=lpb.LPB_SCHED_STREAMED))
    for key in ("status", "iters", "obj", "x", "y"):
        np.testing.assert_array_equal(got[key], want[key], err_msg=key)


@pytest.mark.parametrize("most", ["small", "large"])
def test_every_size_in_either_code(most):
    """The largest one-warp LPs in a batch of small ones and the other way round."""
    counts = (60, 9) if most == "small" else (9, 60)
    lps = [W.mixed_sign_dense(counts[0], 20, 30, start=3).lp(k) for k in range(counts[0])]
    lps += [W.mixed_sign_dense(counts[1], 80, 86, start=4, p_phase1=0.0).lp(k) for k in range(counts[1])]
    batch = W.pack(most, lps)
    got = gpu_solve(batch, opts=lpb.lpb_default_opts(precision=lpb.LP_PREC_FP32_REFINE))
    want = gpu_solve(batch, opts=lpb.lpb_default_opts(precision=lpb.LP_PREC_FP32_REFINE,
                                                      schedule=lpb.LPB_SCHED_STREAMED))
    for key in ("status", "iters", "obj", "x", "y"):
        np.testing.assert_array_equal(got[key], want[key], err_msg=key)


def test_the_line_is_between_the_groups():
    sizes = []
    for m, n in ((50, 50), (62, 40)):
        s = lpb.BatchSolver(W.mixed_sign_dense(60, m, n, start=5, p_phase1=0.4),
                            opts=lpb.lpb_default_opts(precision=lpb.LP_PREC_FP32_REFINE))
        try:
            sizes += [g["smem_bytes"] for g in lpb.lp_batch_groups(s.h) if g["kind"] == 0 and g["threads"] == 32]
        finally:
            s.close()
    assert min(sizes) <= 14 * 1024 < max(sizes), sizes
