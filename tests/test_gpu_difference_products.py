"""The difference-product slice GEMM (256 x 256 C tiles on CTA pairs): results
bit-identical to the oracle's emulation, which takes the digit products one
by one.  Sizes at the edges of its rules: one row, column or k past a tile,
odd tile-row and tile-column counts (a CTA of a pair without a tile), one
k-block, several FP32 windows, tiles cut by segments and by ranges of k, whole
waves with a cut rest; every slice count it takes."""
import ctypes

import numpy as np
import pytest
import torch

import oracle
from paper_1211_1581_gb300 import inputs, mxm
from helpers import assert_bitwise

pytestmark = pytest.mark.gpu


def _emulated(A, B, mode, S):
    if mode == mxm.MODE_EMUL_RN8:
        return oracle.ozaki_gemm_rn8(A, B, S)
    return oracle.ozaki_gemm(A, B, S=S, beta=7 if mode == mxm.MODE_EMUL_I8 else 8)


@pytest.mark.parametrize("mode,S,m,k,n", [
    (mxm.MODE_EMUL_I8, 7, 256, 128, 256),      # one tile, one k-block
    (mxm.MODE_EMUL_I8, 7, 129, 129, 129),      # a second tile row, column, k-block of one
    (mxm.MODE_EMUL_I8, 8, 385, 1040, 257),     # odd tile counts; 9 k-blocks: two windows
    (mxm.MODE_EMUL_I8, 3, 300, 200, 257),
    (mxm.MODE_EMUL_I8, 7, 100, 300, 77),       # a single tile-row and tile-column
    (mxm.MODE_EMUL_RN8, 6, 90, 1000, 600),
    (mxm.MODE_EMUL_BF16, 6, 700, 260, 128),
    (mxm.MODE_EMUL_I8, 4, 260, 300, 513),
    (mxm.MODE_EMUL_I8, 5, 513, 17, 300),
    (mxm.MODE_EMUL_I8, 6, 257, 2100, 130),     # few tiles: cut along k too
    (mxm.MODE_EMUL_I8, 9, 300, 260, 300),
    (mxm.MODE_EMUL_BF16, 3, 200, 300, 200),
    (mxm.MODE_EMUL_BF16, 6, 300, 1777, 257),   # windows of two k-blocks
    (mxm.MODE_EMUL_BF16, 8, 257, 400, 513),
    (mxm.MODE_EMUL_BF16, 6, 257, 6000, 300),   # sums beyond int32: k in ranges
    (mxm.MODE_EMUL_I8, 7, 130, 20000, 257),
    (mxm.MODE_EMUL_RN8, 3, 129, 100, 257),
    (mxm.MODE_EMUL_RN8, 6, 385, 1300, 300),
    (mxm.MODE_EMUL_RN8, 7, 300, 140, 300),
])
def test_bit_identical_to_oracle(mode, S, m, k, n):
    A, B = inputs.gemm_operands("spread", m, k, n, seed=S, cfg=41)
    C = torch.full((m, n), float("nan"), dtype=torch.float64, device="cuda")
    mxm.mxm_gemm(mode, torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda(), C, slices=S)
    assert mxm.mxm_get_device_status() == mxm.MXM_OK
    assert_bitwise(C.cpu().numpy(), _emulated(A, B, mode, S), f"mode {mode} S={S} {m}x{k}x{n}")


@pytest.mark.parametrize("m,k,n,raster", [(2300, 200, 2300, 0), (2300, 200, 2300, 3),
                                          (5000, 130, 4870, 0)])
def test_many_tiles_match_the_products_one_by_one(m, k, n, raster):
    """More tiles than CTA pairs (81 and 380 on 76): whole waves and the cut
    rest, against the single-CTA kernel, which takes no difference products,
    and on sampled entries against the oracle."""
    A, B = inputs.gemm_operands("spread", m, k, n, seed=2, cfg=42)
    dA, dB = torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda()
    C = torch.full((m, n), float("nan"), dtype=torch.float64, device="cuda")
    D = torch.full((m, n), float("nan"), dtype=torch.float64, device="cuda")
    mxm.mxm_gemm_plan(mxm.MODE_EMUL_I8, dA, dB, C, slices=7, plan=mxm.Plan(raster, 0, 0, 0))
    mxm.mxm_gemm_plan(mxm.MODE_EMUL_I8, dA, dB, D, slices=7, plan=mxm.Plan(0, 0, 1, 1))
    assert mxm.mxm_get_device_status() == mxm.MXM_OK
    assert torch.equal(C, D)
    rng = np.random.default_rng(m + raster)
    ii, jj = rng.integers(0, m, 200), rng.integers(0, n, 200)
    assert_bitwise(C.cpu().numpy()[ii, jj], oracle.ozaki_entries(A, B, ii, jj, S=7, beta=7),
                   "sampled entries")


@pytest.mark.parametrize("mode,S,m,k,n", [
    (mxm.MODE_EMUL_I8, 7, 1300, 100, 1050),    # 256 x 128 tiles: 54, one wave, odd tile-rows
    (mxm.MODE_EMUL_I8, 3, 1281, 384, 1025),
    (mxm.MODE_EMUL_I8, 6, 2600, 257, 1100),    # 99: a second wave
    (mxm.MODE_EMUL_RN8, 6, 1290, 300, 1100),   # several windows a segment
    (mxm.MODE_EMUL_BF16, 6, 1300, 1000, 1030),
    (mxm.MODE_EMUL_RN8, 7, 2050, 129, 2050),
])
def test_little_k(mode, S, m, k, n):
    A, B = inputs.gemm_operands("spread", m, k, n, seed=4, cfg=44)
    dA, dB = torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda()
    C = torch.full((m, n), float("nan"), dtype=torch.float64, device="cuda")
    D = torch.full((m, n), float("nan"), dtype=torch.float64, device="cuda")
    mxm.mxm_gemm(mode, dA, dB, C, slices=S)
    mxm.mxm_gemm_plan(mode, dA, dB, D, slices=S, plan=mxm.Plan(0, 0, 1, 1))
    assert mxm.mxm_get_device_status() == mxm.MXM_OK
    assert torch.equal(C, D)
    rng = np.random.default_rng(m)
    ii, jj = rng.integers(0, m, 60), rng.integers(0, n, 60)
    ii[0], jj[0] = m - 1, n - 1
    # an entry depends on its row of A and its column of B alone
    want = np.diagonal(_emulated(A[ii], B[:, jj], mode, S))
    assert_bitwise(C.cpu().numpy()[ii, jj], want, "sampled entries")


def test_smaller_caller_workspace_takes_the_products_one_by_one():
    """A caller workspace of the size the products one by one need (what
    mxm_workspace_size gives under a single-CTA plan) still runs, with the same
    bits; one byte less is refused."""
    m, k, n = 600, 300, 600
    A, B = inputs.gemm_operands("spread", m, k, n, seed=3, cfg=43)
    dA, dB = torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda()
    less = mxm.mxm_workspace_size_plan(mxm.MODE_EMUL_I8, m, k, n, 7, mxm.Plan(0, 0, 1, 0))
    full = mxm.mxm_workspace_size(mxm.MODE_EMUL_I8, m, k, n, 7)
    assert 0 < less < full
    want = oracle.ozaki_gemm(A, B, S=7, beta=7)
    ws = torch.empty(full, dtype=torch.uint8, device="cuda")
    lib = mxm.load()
    try:
        for size, status in ((full, mxm.MXM_OK), (full - 1, mxm.MXM_OK), (less, mxm.MXM_OK),
                             (less - 1, mxm.MXM_ERR_WORKSPACE_TOO_SMALL)):
            assert lib.mxm_set_workspace(ws.data_ptr(), size, None) == mxm.MXM_OK
            C = torch.full((m, n), 7.0, dtype=torch.float64, device="cuda")
            torch.cuda.synchronize()
            st = lib.mxm_gemm(mxm.MODE_EMUL_I8, ctypes.c_void_p(dA.data_ptr()),
                              ctypes.c_void_p(dB.data_ptr()), ctypes.c_void_p(C.data_ptr()),
                              m, k, n, 7, None)
            assert st == status
            torch.cuda.synchronize()
            if st == mxm.MXM_OK:
                assert_bitwise(C.cpu().numpy(), want, f"workspace {size}")
            else:
                assert torch.all(C == 7.0)
    finally:
        torch.cuda.synchronize()
        mxm.mxm_set_workspace(None)


@pytest.mark.parametrize("m,k,n", [(1, 1, 1), (64, 64, 64), (128, 128, 128), (129, 128, 128),
                                   (128, 127, 129), (4096, 64, 64), (100, 30, 4096),
                                   (4097, 64, 64)])
@pytest.mark.parametrize("mode,S", [(mxm.MODE_EMUL_I8, 3), (mxm.MODE_EMUL_I8, 7),
                                    (mxm.MODE_EMUL_BF16, 8), (mxm.MODE_EMUL_RN8, 6)])
def test_one_block_of_one_tile_row_or_column(mode, S, m, k, n):
    """Up to 16 tiles the library's own workspace takes the difference products,
    a caller's of the size it was told takes the digit products one by one, as
    does a single-CTA plan: the same bits."""
    A, B = inputs.gemm_operands("spread", m, k, n, seed=5, cfg=71)
    a, b = torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda()
    outs = [torch.full((m, n), float("nan"), dtype=torch.float64, device="cuda")
            for _ in range(3)]
    mxm.mxm_gemm(mode, a, b, outs[0], slices=S)
    mxm.mxm_gemm_plan(mode, a, b, outs[1], slices=S, plan=mxm.Plan(cta=1))
    ws = torch.empty(mxm.mxm_workspace_size(mode, m, k, n, S), dtype=torch.uint8, device="cuda")
    mxm.mxm_set_workspace(ws)
    try:
        mxm.mxm_gemm(mode, a, b, outs[2], slices=S)
        torch.cuda.synchronize()
    finally:
        mxm.mxm_set_workspace(None)
    assert mxm.mxm_get_device_status() == mxm.MXM_OK
    assert torch.equal(outs[0], outs[1]) and torch.equal(outs[0], outs[2])
