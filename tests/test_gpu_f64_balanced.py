"""Native FP64 in equal shares: sizes at the edges of its pieces (32 x 32 cut
into m16 / n8 DMMA blocks, steps of 4 k), products of less than a step per
share, k too short to be cut, the plan's k ranges, and a caller workspace too
small for all shares.  Against the Dot2 oracle within 2 k u |A||B|, and
bit-exact on small integers."""
import numpy as np
import pytest
import torch

import oracle
from paper_1211_1581_gb300 import inputs, mxm
from helpers import assert_bitwise, assert_within_bound

pytestmark = pytest.mark.gpu

SHAPES = [(1, 1, 1), (1, 32, 1), (16, 33, 8), (17, 31, 9), (32, 64, 32), (33, 65, 41),
          (48, 127, 72), (100, 3, 100), (64, 1000, 17), (300, 33, 17), (257, 129, 263),
          (15, 5000, 7), (700, 40, 650)]


def _product(A, B, plan=None):
    C = torch.full((A.shape[0], B.shape[1]), float("nan"), dtype=torch.float64, device="cuda")
    mxm.mxm_gemm_plan(mxm.MODE_F64, torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda(), C, 0,
                      plan)
    assert mxm.mxm_get_device_status() == mxm.MXM_OK
    return C.cpu().numpy()


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("splitk", [0, 1, 3])
def test_within_bound_and_exact_on_integers(shape, splitk):
    m, k, n = shape
    plan = mxm.Plan(0, 0, 0, splitk)
    A, B = inputs.gemm_operands("spread", m, k, n, seed=5, cfg=51)
    got = _product(A, B, plan)
    assert_within_bound(got, oracle.gemm_dot2(A, B), oracle.gemm_abs(A, B), k, f"{shape}")
    A, B = inputs.gemm_operands("int8", m, k, n, seed=5, cfg=52)
    assert_bitwise(_product(A, B, plan), oracle.gemm_dot2(A, B), f"{shape} integers")


def test_smaller_caller_workspace_cuts_fewer_shares():
    """The size held before the shares existed (here 2 MiB: room for 127 of the
    1216 shares) still runs; one byte less than it is refused."""
    m = k = n = 256
    least = (2 + 2) * 16 * 16384 + 2 * 4 * 128 * 128 * 8
    assert mxm.mxm_workspace_size(mxm.MODE_F64, m, k, n) > least
    A, B = inputs.gemm_operands("int8", m, k, n, seed=6, cfg=53)
    want = oracle.gemm_dot2(A, B)
    ws = torch.empty(least, dtype=torch.uint8, device="cuda")
    try:
        mxm.mxm_set_workspace(ws)
        assert_bitwise(_product(A, B), want, "fewer shares")
        mxm.mxm_set_workspace(ws[:least - 1])
        with pytest.raises(mxm.MxmError) as ei:
            _product(A, B)
        assert ei.value.status == mxm.MXM_ERR_WORKSPACE_TOO_SMALL
    finally:
        torch.cuda.synchronize()
        mxm.mxm_set_workspace(None)
    assert np.array_equal(_product(A, B), want)
