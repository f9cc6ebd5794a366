"""The conjugate-gradient engine over all SMs on matrices whose rows differ
much in length: long rows that are neighbours, in front, at the end and inside,
so that the rows are cut by work.  Against the oracle, with the tolerances of
test_gpu_cg; and the same bits every time."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
from paper_1211_1581_gb300 import mxm  # noqa: E402
from test_gpu_cg import compare, run_cg  # noqa: E402

pytestmark = pytest.mark.gpu


def coupled(n, sets, seed=1):
    """Symmetric, strictly diagonally dominant CSR: neighbours coupled, and the
    rows of every index set in `sets` all coupled with each other."""
    rng = np.random.default_rng(seed)
    i = np.arange(n - 1)
    c = rng.uniform(-0.3, 0.3, n - 1)
    rows, cols, vals = [i, i + 1, np.arange(n)], [i + 1, i, np.arange(n)], [c, c, np.full(n, 5.0)]
    for s in sets:
        s = np.asarray(s, dtype=np.int64)
        a = rng.uniform(-1, 1, (len(s), len(s))) / len(s)
        a = a + a.T
        r, q = np.meshgrid(s, s, indexing="ij")
        keep = np.abs(r - q) > 1
        rows.append(r[keep])
        cols.append(q[keep])
        vals.append(a[keep])
    r, c, v = np.concatenate(rows), np.concatenate(cols), np.concatenate(vals)
    o = np.argsort(r * n + c, kind="stable")
    rowp = np.zeros(n + 1, dtype=np.int64)
    rowp[1:] = np.cumsum(np.bincount(r, minlength=n))
    return rowp.astype(np.int32), c[o].astype(np.int32), v[o]


NEIGHBOURS = {
    "front": (30000, lambda n: [np.arange(400)]),
    "end": (200000, lambda n: [np.arange(n - 658, n)]),
    "inside, twice": (160000, lambda n: [np.arange(70000, 70300), np.arange(140000, 140500)]),
    "few rows": (300, lambda n: [np.arange(100, 250)]),
}


def check(rowp, indx, vals, longest):
    n = len(rowp) - 1
    b = np.random.default_rng(n).uniform(-1, 1, n)
    stop = 1e-24 * float(b @ b)
    got, _ = compare(rowp, indx, vals, b, stop, 200, longest, mxm.CG_GRAPH)
    assert got["iters"] > 5
    again = run_cg(rowp, indx, vals, b, stop, 200, engine=mxm.CG_GRAPH)
    assert np.array_equal(got["x"], again["x"]) and got["r2"] == again["r2"]


@pytest.mark.parametrize("case", list(NEIGHBOURS))
def test_long_rows_beside_each_other(case):
    n, sets = NEIGHBOURS[case]
    rowp, indx, vals = coupled(n, sets(n))
    check(rowp, indx, vals, int(np.diff(rowp).max()))
