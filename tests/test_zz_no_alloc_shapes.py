"""lp_solve_uniform_noalloc on shapes at which its choice of kernel differs from
the regular plan's (it knows neither the number of artificials nor the sign of
A), against the regular entry point bit for bit."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


# e = (m + 1)(n + m + 1) around 14,000 entries: tall, square, wide, rows beyond 1024 entries, one row
@pytest.mark.parametrize("m,n", [(120, 20), (110, 15), (83, 83), (84, 83), (30, 420), (8, 1600), (1, 6998), (1, 6999),
                                 (130, 130), (20, 1100)])
@pytest.mark.parametrize("signed", [False, True])
def test_shapes(m, n, signed):
    import torch
    from paper_1802_08557_gb300 import build, lpbatch as lpb
    from paper_1802_08557_gb300 import workloads as W
    build.build()
    lpb.load()
    g = np.random.default_rng(m * 20011 + n)
    lo, N = -1 if signed else 0, 7
    lps = [(g.uniform(lo, 1, (m, n)), g.uniform(-2 if signed else 1, 10, m), g.uniform(lo, 1, n)) for _ in range(N)]
    batch = W.pack("shapes", lps)
    s = lpb.BatchSolver(batch, device_data=True)
    try:
        s.solve()
        ref = s.results()
    finally:
        s.close()
    dev = torch.device("cuda")
    A, b, c = (torch.from_numpy(v).to(dev) for v in (batch.A, batch.b, batch.c))
    status, iters = (torch.full((N,), -7, dtype=torch.int32, device=dev) for _ in range(2))
    obj, x, y = (torch.full((k,), float("nan"), dtype=torch.float64, device=dev) for k in (N, N * n, N * m))
    rc = lpb.lp_solve_uniform_noalloc(N, m, n, A, b, c, status, iters, obj, x, y, None, torch.cuda.current_stream())
    assert rc == lpb.LPB_OK
    torch.cuda.synchronize()
    for name, t in (("status", status), ("iters", iters), ("obj", obj), ("x", x), ("y", y)):
        np.testing.assert_array_equal(t.cpu().numpy(), ref[name], err_msg=name)
