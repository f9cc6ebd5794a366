"""Split-k partial sums of the digit products: int32 up to the largest k range
whose diagonal sums fit (43 k-blocks of 8-bit digits at S = 6, every digit at
its largest), int64 from the next k-block on; both give the bits of the
unsplit product."""
import pytest
import torch

from paper_1211_1581_gb300 import mxm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("blocks", [43, 44])
@pytest.mark.parametrize("splits", [2, 33])  # a thread for all ranges, eight threads
@pytest.mark.parametrize("largest", [True, False])
def test_partials_at_the_edge_of_int32(blocks, splits, largest):
    m, n, k = 40, 136, 128 * blocks * splits
    if largest:  # digits of 1 - 2^-53: all 255
        A = torch.full((m, k), 1.0 - 2.0 ** -53, dtype=torch.float64, device="cuda")
        B = torch.full((k, n), -(1.0 - 2.0 ** -53), dtype=torch.float64, device="cuda")
    else:
        g = torch.Generator(device="cuda")
        g.manual_seed(blocks)
        A = torch.rand((m, k), dtype=torch.float64, device="cuda", generator=g) - 0.5
        B = torch.rand((k, n), dtype=torch.float64, device="cuda", generator=g) - 0.5
    split = torch.full((m, n), float("nan"), dtype=torch.float64, device="cuda")
    whole = torch.full((m, n), float("nan"), dtype=torch.float64, device="cuda")
    mxm.mxm_gemm_plan(mxm.MODE_EMUL_BF16, A, B, split, slices=6, plan=mxm.Plan(splitk=splits))
    mxm.mxm_gemm_plan(mxm.MODE_EMUL_BF16, A, B, whole, slices=6, plan=mxm.Plan(cta=1, splitk=1))
    torch.cuda.synchronize()
    assert mxm.mxm_get_device_status() == mxm.MXM_OK
    assert torch.equal(split, whole)
