"""Split-k products of few rows, whose fold is launched after the slice GEMM,
and of more, whose fold is launched beside it: the bits of the oracle's
emulation, also back to back; and few rows take no longer than sixteen, which do
the same work."""
import numpy as np
import pytest
import torch

import oracle
from paper_1211_1581_gb300 import inputs, mxm
from helpers import assert_bitwise

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,k,n", [(1, 2000, 1500), (1, 20000, 40), (15, 1100, 300), (16, 1100, 300),
                                   (7, 40000, 5), (1, 9000, 1)])
def test_bits(m, k, n):
    A, B = inputs.gemm_operands("spread", m, k, n, seed=9, cfg=91)
    a, b = torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda()
    outs = [torch.full((m, n), float("nan"), dtype=torch.float64, device="cuda") for _ in range(4)]
    for c in outs:
        mxm.mxm_f64_emul(a, b, c, 7)
    assert mxm.mxm_get_device_status() == mxm.MXM_OK
    assert_bitwise(outs[0].cpu().numpy(), oracle.ozaki_gemm(A, B, S=7, beta=7), f"{m}x{k}x{n}")
    assert all(torch.equal(c, outs[0]) for c in outs)


def test_one_row_takes_no_longer_than_sixteen():
    def median(m):
        a = torch.rand((m, 4096), dtype=torch.float64, device="cuda") - 0.5
        b = torch.rand((4096, 4096), dtype=torch.float64, device="cuda") - 0.5
        c = torch.empty((m, 4096), dtype=torch.float64, device="cuda")
        times = []
        for i in range(14):
            e0, e1 = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            e0.record()
            mxm.mxm_f64_emul(a, b, c, 7)
            e1.record()
            torch.cuda.synchronize()
            if i >= 3:
                times.append(e0.elapsed_time(e1))
        return np.median(times)

    assert median(1) < 1.2 * median(16)
