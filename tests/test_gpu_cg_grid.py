"""The conjugate-gradient engine over all SMs at the edges of its layout: one
lane a row up to a whole warp a row, fewer rows than blocks, vectors in shared
memory and (beyond 1.4 million rows) in global memory, rows of very uneven
length, and no step at all.  Against the oracle, with the tolerances of
test_gpu_cg."""
import numpy as np
import pytest

from paper_1211_1581_gb300 import inputs

torch = pytest.importorskip("torch")
from paper_1211_1581_gb300 import mxm  # noqa: E402
from test_gpu_cg import compare, run_cg  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,bw", [(100, 3), (152, 31), (3000, 65), (12000, 33), (40000, 9),
                                  (90000, 5), (200000, 3), (160000, 17), (1500000, 3)])
def test_lanes_per_row_and_layout(n, bw):
    rowp, indx, vals = inputs.banded_spd(31, 122, n, bw)
    b = inputs.uniform_pm1(31, 123, (n,))
    got, _ = compare(rowp, indx, vals, b, 1e-20 * float(b @ b), 100, bw, mxm.CG_GRAPH)
    assert got["iters"] > 5


def test_uneven_rows():
    """A diagonal matrix bordered by one full row and column: rows of 2 values
    beside one of n."""
    n = 5000
    rng = np.random.default_rng(3)
    c = rng.uniform(-1, 1, n - 1) / n
    rowp = np.concatenate(([0, n], n + 2 * np.arange(1, n))).astype(np.int32)
    indx = np.empty(rowp[-1], dtype=np.int32)
    vals = np.empty(rowp[-1])
    indx[:n] = np.arange(n)
    vals[:n] = np.concatenate(([4.0], c))
    indx[n::2], indx[n + 1::2] = 0, np.arange(1, n)
    vals[n::2], vals[n + 1::2] = c, 2.0 + rng.uniform(0, 1, n - 1)
    b = rng.uniform(-1, 1, n)
    compare(rowp, indx, vals, b, 1e-24 * float(b @ b), 200, n, mxm.CG_GRAPH)


def test_no_step():
    rowp, indx, vals = inputs.banded_spd(32, 124, 20000, 5)
    b = inputs.uniform_pm1(32, 125, (20000,))
    for stop, most in ((2.0 * float(b @ b), 10), (0.0, 0)):
        got = run_cg(rowp, indx, vals, b, stop, most, engine=mxm.CG_GRAPH)
        assert got["iters"] == 0 and np.all(got["x"] == 0.0)
        assert abs(got["r2"] - float(b @ b)) <= 1e-12 * float(b @ b)
