"""FP64 deferred updates of large LPs, the forms that a batch reaches only by
size or number: the 256-thread class of packing LPs by the thousand, with LPs
that are taken for packing LPs and are not (flushes, phase I), and vectors that
exceed one CTA's shared memory; against the oracle bit for bit."""
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


def _looked_at(size):
    """The entries of A that the FP64 plan reads: 4 in a row at 64 places."""
    i = np.arange(256)
    return i // 4 * (size - 4) // 63 + i % 4


def _dense(m, n, seed, signed=False, phase1=False, hidden=False):
    g = np.random.default_rng(seed)
    A = g.uniform(-1 if signed else 0, 1, (m, n))
    b = g.uniform(1, 10 if signed else 100, m)
    if phase1:
        b[3::7] = -g.uniform(0.1, 2, len(b[3::7]))
    if hidden:
        at = _looked_at(m * n)
        A.reshape(-1)[at] = np.abs(A.reshape(-1)[at])
    return A, b, g.uniform(-1 if signed else 0, 1, n)


def _repeated(lps, count):
    p = W.pack("kinds", lps)
    rep = lambda v: np.repeat(v, count)
    return p, W.LPBatch("repeated", rep(p.m), rep(p.n), rep(p.a_off), rep(p.b_off), rep(p.c_off), p.A, p.b, p.c)


def test_packing_class_with_wrong_guesses():
    import torch
    lps = [_dense(300, 290, 1), _dense(64, 900, 2), _dense(900, 64, 3),
           _dense(270, 60, 4, signed=True, hidden=True), _dense(60, 270, 5, signed=True, hidden=True),
           _dense(260, 90, 6, signed=True, phase1=True, hidden=True),
           _dense(90, 260, 7, signed=True, phase1=True, hidden=True)]
    count = 16 * torch.cuda.get_device_properties(0).multi_processor_count // len(lps) + 1
    p, batch = _repeated(lps, count)
    s = lpb.BatchSolver(batch)
    try:
        groups = lpb.lp_batch_groups(s.h)
        assert [(g["kind"], g["threads"]) for g in groups] == [(2, 256)], groups
    finally:
        s.close()
    got = gpu_solve(batch)
    ref = oracle_solve(p)
    # more pivots than are kept pending before a flush: half of m w / (m + w), at least 16
    for k in (3, 4, 5, 6):
        m, w = int(p.m[k]), int(p.n[k]) + int((lps[k][1] < 0).sum()) + 1
        assert ref["iters"][k] > max(16, m * w // (2 * (m + w))), (k, ref["iters"][k])
    first = np.arange(len(lps)) * count
    assert compare(batch, got, ref, idx=first) == (len(lps), len(lps))
    # every copy has its first one's outputs
    assert (got["iters"].reshape(-1, count) == got["iters"][first][:, None]).all()
    assert (got["obj"].reshape(-1, count) == got["obj"][first][:, None]).all()


def test_fewer_packing_lps_take_512_threads():
    s = lpb.BatchSolver(_repeated([_dense(300, 290, 1)], 600)[1])
    try:
        assert [(g["kind"], g["threads"]) for g in lpb.lp_batch_groups(s.h)] == [(2, 512)]
    finally:
        s.close()


def _vector_bytes(m, n):
    """Per-row and per-column vectors of an LP with every row negated."""
    up = lambda v: -(-v // 16) * 16
    w = n + m + 1
    return up(8 * m) + 5 * up(4 * m) + 2 * up(8 * w) + 2 * up(4 * w)


CTA_BYTES = 227 * 1024 - 1024 - 640


@pytest.mark.parametrize("m,n,signed,phase1", [(40, 9700, False, False), (12, 10500, True, False),
                                               (12, 10500, False, True), (30, 12000, True, True)])
def test_vectors_in_the_workspace(m, n, signed, phase1):
    assert _vector_bytes(m, n) > CTA_BYTES
    batch = W.pack("wide", [_dense(m, n, m + n, signed=signed, phase1=phase1)])
    got = gpu_solve(batch)
    assert got["plan"]["num_streamed"] == 1
    assert compare(batch, got, oracle_solve(batch)) == (1, 1)


# one row or column past each class's threads, and the last within them
@pytest.mark.parametrize("edge", [32, 64, 128, 256, 1024])
def test_class_edges(edge):
    lps = []
    for d in (edge - 1, edge, edge + 1):  # d = columns + 1, or rows
        lps += [_dense(17, d - 1, d, signed=True), _dense(d, 15, d, signed=True), _dense(19, d - 4, d, phase1=True)]
    batch = W.pack("edges", lps)
    got = gpu_solve(batch, opts=lpb.lpb_default_opts(schedule=lpb.LPB_SCHED_STREAMED))
    assert got["plan"]["num_streamed"] == len(lps)
    assert compare(batch, got, oracle_solve(batch)) == (len(lps), len(lps))


# several threads per column in a flush: columns that divide the group's threads and that do not, rows left
# over, retired columns (phase I)
@pytest.mark.parametrize("phase1", [False, True])
def test_flushes_of_few_columns(phase1):
    sizes = [(225, 64), (250, 40), (128, 25), (120, 20), (63, 21), (250, 85), (200, 50), (97, 32)]
    lps = [_dense(m, n, 31 * m + n, signed=True, phase1=phase1) for m, n in sizes]
    batch = W.pack("tall", lps)
    ref = oracle_solve(batch)
    pending = [max(16, m * (n + 1) // (2 * (m + n + 1))) for m, n in sizes]
    if not phase1:
        assert all(it > p for it, p in zip(ref["iters"], pending)), (list(ref["iters"]), pending)
    got = gpu_solve(batch, opts=lpb.lpb_default_opts(schedule=lpb.LPB_SCHED_STREAMED))
    assert got["plan"]["num_streamed"] == len(lps)
    assert compare(batch, got, ref) == (len(lps), len(lps))
