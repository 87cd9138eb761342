"""Hyperbox LPs at the row lengths where the tile kernel changes its form: 1, 2
or 4 coordinates per step, each bank-swap rule (dim a multiple of 4, 8, 16), the
line between tiles of 128 and of 32, and numbers of LPs around a tile; and above
64 coordinates several LPs per warp with a last warp of every fill.  Integer
data: every sum is exact, so objectives match the oracle bit for bit in any order
of the FMAs, and a coordinate paired with another's bound shows."""
import numpy as np
import pytest

from oracle import hyperbox as ohb
from paper_1802_08557_gb300 import lpbatch as lpb

pytestmark = pytest.mark.gpu


def _check(num, dim, per_lp):
    import torch
    g = np.random.default_rng(1000 * dim + 2 * num + per_lp)
    L = g.integers(-1000, 1001, (num, dim)).astype(np.float64)
    L[g.random((num, dim)) < 0.1] = -0.0
    shape = (num, dim) if per_lp else (dim,)
    lo = g.integers(-1000, 1, shape).astype(np.float64)
    hi = lo + g.integers(0, 1000, shape)
    want_obj, want_x = ohb.hyperbox_solve(L, lo, hi)
    dL, dlo, dhi = (torch.from_numpy(a).cuda() for a in (L, lo, hi))
    obj, x = torch.empty(num, dtype=torch.float64, device="cuda"), torch.empty_like(dL)
    lpb.lp_hyperbox_solve(dL, dlo, dhi, obj, x, box_per_lp=per_lp, ptr_kind=lpb.LPB_DEVICE,
                          stream=torch.cuda.current_stream())
    torch.cuda.synchronize()
    np.testing.assert_array_equal(obj.cpu().numpy(), want_obj)
    np.testing.assert_array_equal(x.cpu().numpy(), want_x)


@pytest.mark.parametrize("per_lp", [False, True])
@pytest.mark.parametrize("dim", [3, 4, 6, 8, 9, 10, 12, 13, 16, 20, 24, 40, 48, 62, 64])
def test_row_forms_match_the_oracle(dim, per_lp):
    for num in (1, 31, 33, 128, 397):
        _check(num, dim, per_lp)


@pytest.mark.parametrize("per_lp", [False, True])
@pytest.mark.parametrize("num", range(20000, 20008))
def test_several_lps_per_warp_match_the_oracle(num, per_lp):
    _check(num, 65 + num % 8 * 13, per_lp)
