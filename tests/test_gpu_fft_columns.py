"""The transform's pass and cluster kernels at every order, with tables of the
order itself and of larger ones, on inputs with signed zeros: the results do not
depend on the table's order, and match numpy's transform within the radix-2
bound."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
from paper_1211_1581_gb300 import inputs, mxm  # noqa: E402

pytestmark = pytest.mark.gpu
U = 2.0 ** -53


@pytest.mark.parametrize("p", [1, 2, 3, 4, 5, 7, 8, 11, 13, 14, 15, 16, 17, 19, 20, 21, 22])
def test_orders_and_tables(p):
    n = 1 << p
    v = inputs.uniform_pm1(p, 170, (2 * n,))
    v[::7] = -0.0
    x = torch.from_numpy(v).cuda().view(torch.complex128)
    got = mxm.FFT(n)(x)
    lib = mxm.load()
    big = min(4 * n, lib.mxm_fft_max_n())
    f = mxm.FFT(big)
    other, work = torch.empty_like(x), torch.empty_like(x)
    st = lib.mxm_fft(x.data_ptr(), other.data_ptr(), work.data_ptr(), f.table.data_ptr(), big, n,
                     torch.cuda.current_stream().cuda_stream)
    assert st == mxm.MXM_OK
    assert torch.equal(torch.view_as_real(got), torch.view_as_real(other))
    want = np.fft.fft(v.view(complex))
    err = np.linalg.norm(got.cpu().numpy() - want)
    assert err <= 2 * (p + 1) * 8 * U * np.linalg.norm(want)
