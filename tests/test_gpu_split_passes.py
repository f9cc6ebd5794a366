"""The scale and split passes at the edges of their layouts, through whole
products bit-identical to the oracle: rows shared 8, 4, 2 and 1 to a block, rows
too long for the fused pass (their maxima in runs of 2048), every digit kind
with and without difference planes, and wide ranges of exponents (digits cut
off at both ends of the word)."""
import numpy as np
import pytest
import torch

import oracle
from paper_1211_1581_gb300 import inputs, mxm
from helpers import assert_bitwise

pytestmark = pytest.mark.gpu


def _run(mode, A, B, S):
    C = torch.full((A.shape[0], B.shape[1]), float("nan"), dtype=torch.float64, device="cuda")
    mxm.mxm_gemm(mode, torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda(), C, slices=S)
    assert mxm.mxm_get_device_status() == mxm.MXM_OK
    want = (oracle.ozaki_gemm_rn8(A, B, S) if mode == mxm.MODE_EMUL_RN8 else
            oracle.ozaki_gemm(A, B, S=S, beta=7 if mode == mxm.MODE_EMUL_I8 else 8))
    assert_bitwise(C.cpu().numpy(), want, f"mode {mode} S={S} {A.shape} {B.shape}")


@pytest.mark.parametrize("mode,S", [(mxm.MODE_EMUL_I8, 1), (mxm.MODE_EMUL_I8, 2),
                                    (mxm.MODE_EMUL_I8, 9), (mxm.MODE_EMUL_I8, 10),
                                    (mxm.MODE_EMUL_BF16, 1), (mxm.MODE_EMUL_BF16, 8),
                                    (mxm.MODE_EMUL_BF16, 9), (mxm.MODE_EMUL_RN8, 1),
                                    (mxm.MODE_EMUL_RN8, 2), (mxm.MODE_EMUL_RN8, 7)])
@pytest.mark.parametrize("k", [100, 257, 600, 1100])
def test_rows_per_block_and_digit_kinds(mode, S, k):
    rng = np.random.default_rng(k + S)
    A = rng.standard_normal((131, k)) * np.exp2(rng.integers(-70, 70, (131, k)).astype(float))
    B = rng.standard_normal((k, 130)) * np.exp2(rng.integers(-70, 70, (k, 130)).astype(float))
    A[3], B[:, 5], A[7, 3] = 0.0, 0.0, 2.0 ** -1060
    _run(mode, A, B, S)


@pytest.mark.parametrize("k", [24576, 24577, 26625])
def test_long_rows(k):
    A, B = inputs.gemm_operands("spread", 20, k, 9, seed=8, cfg=61)
    A[4, :] = 0.0
    A[5, :-1] = 0.0   # the maximum in the last run alone
    A[6] *= 2.0 ** -1000
    _run(mxm.MODE_EMUL_I8, A, B, 7)
