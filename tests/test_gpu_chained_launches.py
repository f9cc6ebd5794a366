"""Launches of one call that overlap their predecessor: calls queued back to back
on one stream, each with inputs of its own and all sharing the library's
workspace, give what the same calls give one at a time with a synchronisation
between them, bit for bit; so do replays of a captured sequence, and two streams
at once.  Emulated results are also compared with the entry point that runs
ordinary launches only (mxm_f64_emul_noalloc)."""
import pytest
import torch

from paper_1211_1581_gb300 import mxm

pytestmark = pytest.mark.gpu

CALLS = 12
# one k-block, several, k ranges, rows too long for the fused split, one tile
SHAPES = [(64, 64, 64), (300, 200, 520), (130, 9000, 128), (40, 24600, 72), (700, 300, 1100)]


def _operands(m, k, n):
    g = torch.Generator(device="cuda")
    g.manual_seed(m + k + n)
    A = [torch.rand((m, k), dtype=torch.float64, device="cuda", generator=g) - 0.5
         for _ in range(CALLS)]
    B = [torch.rand((k, n), dtype=torch.float64, device="cuda", generator=g) - 0.5
         for _ in range(CALLS)]
    return A, B


def _outs(m, n):
    return [torch.full((m, n), float("nan"), dtype=torch.float64, device="cuda")
            for _ in range(CALLS)]


@pytest.mark.parametrize("mode,S", [(mxm.MODE_EMUL_I8, 7), (mxm.MODE_EMUL_BF16, 6),
                                    (mxm.MODE_EMUL_RN8, 2), (mxm.MODE_F64, 0)])
@pytest.mark.parametrize("m,k,n", SHAPES)
def test_products_back_to_back(mode, S, m, k, n):
    A, B = _operands(m, k, n)
    alone, queued, captured = _outs(m, n), _outs(m, n), _outs(m, n)
    ws = torch.empty(max(16, mxm.mxm_workspace_size(mode, m, k, n, max(S, 1))),
                     dtype=torch.uint8, device="cuda")
    mxm.mxm_set_workspace(ws)  # a capture allocates nothing
    try:
        for a, b, c in zip(A, B, alone):
            mxm.mxm_gemm(mode, a, b, c, slices=S)
            torch.cuda.synchronize()
        for a, b, c in zip(A, B, queued):
            mxm.mxm_gemm(mode, a, b, c, slices=S)
        torch.cuda.synchronize()
        side = torch.cuda.Stream()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=side):
            for a, b, c in zip(A, B, captured):
                mxm.mxm_gemm(mode, a, b, c, slices=S, stream=side)
        graph.replay()
        graph.replay()
        torch.cuda.synchronize()
    finally:
        mxm.mxm_set_workspace(None)
    assert mxm.mxm_get_device_status() == mxm.MXM_OK
    for one, two, three in zip(alone, queued, captured):
        assert torch.equal(one, two) and torch.equal(one, three)


@pytest.mark.parametrize("m,k,n", [s for s in SHAPES if s[1] < 20000])  # its scratch is fixed
def test_against_ordinary_launches(m, k, n):
    A, B = _operands(m, k, n)
    queued, plain = _outs(m, n), _outs(m, n)
    for a, b, c in zip(A, B, queued):
        mxm.mxm_gemm(mxm.MODE_EMUL_I8, a, b, c, slices=7)
    for a, b, c in zip(A, B, plain):
        mxm.mxm_f64_emul_noalloc(a, b, c, 7)
    torch.cuda.synchronize()
    for one, two in zip(queued, plain):
        assert torch.equal(one, two)


@pytest.mark.parametrize("p", [14, 15, 18])
def test_two_pass_transforms_back_to_back(p):
    g = torch.Generator(device="cuda")
    g.manual_seed(p)
    plan = [mxm.FFT(1 << p) for _ in range(2)]
    x = [torch.view_as_complex(torch.rand((1 << p, 2), dtype=torch.float64, device="cuda",
                                          generator=g)) for _ in range(CALLS)]
    alone, queued = [torch.empty_like(v) for v in x], [torch.empty_like(v) for v in x]
    for v, o in zip(x, alone):
        plan[0](v, o)
        torch.cuda.synchronize()
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]  # a plan (work buffer) for each
    for i, (v, o) in enumerate(zip(x, queued)):
        plan[i & 1](v, o, stream=streams[i & 1])
    torch.cuda.synchronize()
    for one, two in zip(alone, queued):
        assert torch.equal(torch.view_as_real(one), torch.view_as_real(two))
