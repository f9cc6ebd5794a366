"""Native FP64 in the workspace that its kernels use, less than the size of the
tile copies that mxm_workspace_size still gives: the bits of the library's own
workspace; one byte less is refused; and no workspace at all for little k."""
import pytest
import torch

from paper_1211_1581_gb300 import mxm

pytestmark = pytest.mark.gpu

SLOTS = (1216 + 1) * (2 * 32 * 32 * 8 + 16)


def _operands(m, k, n):
    g = torch.Generator(device="cuda")
    g.manual_seed(m + k + n)
    return (torch.rand((m, k), dtype=torch.float64, device="cuda", generator=g) - 0.5,
            torch.rand((k, n), dtype=torch.float64, device="cuda", generator=g) - 0.5,
            torch.full((m, n), float("nan"), dtype=torch.float64, device="cuda"))


@pytest.mark.parametrize("m,k,n,need", [(1024, 700, 1024, SLOTS), (4000, 400, 3000, SLOTS),
                                        (300, 20, 500, 0)])
def test_what_the_kernels_use_is_enough(m, k, n, need):
    assert mxm.mxm_workspace_size(mxm.MODE_F64, m, k, n) > need
    A, B, C = _operands(m, k, n)
    own = mxm.mxm_f64(A, B, C).clone()
    ws = torch.empty(max(need, 1), dtype=torch.uint8, device="cuda")
    try:
        mxm.mxm_set_workspace(ws)
        C.fill_(float("nan"))
        mxm.mxm_f64(A, B, C)
        torch.cuda.synchronize()
        assert torch.equal(C, own)
        if need:
            mxm.mxm_set_workspace(ws[:need - 1])
            with pytest.raises(mxm.MxmError) as ei:
                mxm.mxm_f64(A, B, C)
            assert ei.value.status == mxm.MXM_ERR_WORKSPACE_TOO_SMALL
    finally:
        torch.cuda.synchronize()
        mxm.mxm_set_workspace(None)
    assert mxm.mxm_get_device_status() == mxm.MXM_OK


def test_the_library_allocates_no_more():
    m, k, n = 4000, 1000, 4000
    assert mxm.mxm_workspace_size(mxm.MODE_F64, m, k, n) > 60 << 20
    A, B, C = _operands(m, k, n)
    mxm.mxm_set_workspace(None)
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    mxm.mxm_f64(A, B, C)
    torch.cuda.synchronize()
    assert before - torch.cuda.mem_get_info()[0] <= 32 << 20
