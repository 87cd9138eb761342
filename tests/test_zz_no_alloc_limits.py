"""lp_solve_uniform_noalloc at its scratch limit: the largest LPs that it takes
(square and wide), solved with deferred updates in a workspace slot that is
larger than the tableau that the limit counts, against the regular entry point
bit for bit; one row or column more is refused.

Collected last: these LPs are the slowest of the suite."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

LIMIT = 64 << 20


def _within(m, n):
    """One LP's descriptors (8 arrays of 256 bytes), the counter's 256 and its whole phase-I tableau."""
    up = lambda v, a: -(-v // a) * a
    ld = up(n + m + 1, 4)
    tableau = up(8 * m, 16) + 2 * up(4 * m, 16) + up((m + 2) * ld * 8, 16) + up((m + 2) * 8, 16) + up(4 * ld, 16)
    return 256 + 8 * 256 + up(tableau, 256) <= LIMIT


@pytest.mark.parametrize("square", [True, False])
def test_largest_lps_within_the_scratch(square):
    import torch
    from paper_1802_08557_gb300 import build, lpbatch as lpb
    from paper_1802_08557_gb300 import workloads as W
    build.build()
    lpb.load()
    n_of = (lambda m: m) if square else (lambda m: 16384)
    m = max(k for k in range(1, 4096) if _within(k, n_of(k)))
    n = n_of(m)
    g = np.random.default_rng(m)
    batch = W.pack("limit", [(g.uniform(0, 1, (m, n)), g.uniform(1, 100, m), g.uniform(0, 1, n))])
    s = lpb.BatchSolver(batch, device_data=True)
    try:
        s.solve()
        ref = s.results()
    finally:
        s.close()
    dev = torch.device("cuda")
    A, b, c = (torch.from_numpy(v).to(dev) for v in (batch.A, batch.b, batch.c))
    status, iters = (torch.full((1,), -7, dtype=torch.int32, device=dev) for _ in range(2))
    obj, x, y = (torch.full((k,), float("nan"), dtype=torch.float64, device=dev) for k in (1, n, m))
    out = (status, iters, obj, x, y, None, torch.cuda.current_stream())
    assert lpb.lp_solve_uniform_noalloc(1, m, n, A, b, c, *out) == lpb.LPB_OK
    torch.cuda.synchronize()
    for name, t in (("status", status), ("iters", iters), ("obj", obj), ("x", x), ("y", y)):
        np.testing.assert_array_equal(t.cpu().numpy(), ref[name], err_msg=name)
    # (refused before any pointer is read)
    assert lpb.lp_solve_uniform_noalloc(1, m + 1, n_of(m + 1), A, b, c, *out) == lpb.LPB_ETOOBIG
