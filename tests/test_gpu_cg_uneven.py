"""The conjugate-gradient engine over all SMs on matrices whose rows differ
much in length: long rows that are neighbours, in front, at the end and inside,
so that the rows are cut by work; long rows among short ones, a warp's each; and
full rows, a block's each.  Against the same iteration in extended precision,
with the tolerances of test_gpu_cg (the oracle adds a row of 200,000 values one
by one in FP64 and is itself further off than those allow: r2 of step 12 of a
matrix with three full rows by 6.8e-9 of 4.8e-9, this engine's by 2.3e-10); and
the same bits every time."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
from paper_1211_1581_gb300 import mxm  # noqa: E402
from test_gpu_cg import U, gershgorin, run_cg  # noqa: E402

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


def extended_cg(rowp, indx, vals, b, stop, max_iters):
    """The iteration in long double; every row holds at least its diagonal."""
    v, r = vals.astype(np.longdouble), b.astype(np.longdouble)
    x, p, r2, hist = np.zeros_like(r), r.copy(), np.sum(r * r), []
    while r2 > stop and len(hist) < max_iters:
        q = np.add.reduceat(v * p[indx], rowp[:-1])
        alpha = r2 / np.sum(p * q)
        x += alpha * p
        r -= alpha * q
        r2, old = np.sum(r * r), r2
        p = r + (r2 / old) * p
        hist.append(r2)
    return x.astype(np.float64), np.array(hist, dtype=np.float64)


def check(rowp, indx, vals, longest):
    n = len(rowp) - 1
    b = np.random.default_rng(n).uniform(-1, 1, n)
    stop = 1e-24 * float(b @ b)
    x, h = extended_cg(rowp, indx, vals, b, stop, 200)
    got = run_cg(rowp, indx, vals, b, stop, 200, engine=mxm.CG_GRAPH)
    lo, hi = gershgorin(rowp, indx, vals)
    kap = hi / lo
    assert kap <= 1000 and got["iters"] > 5
    tol = lambda k: 4 * kap * (n + longest) * U * (k + 1)  # noqa: E731
    near = np.any(np.abs(h / stop - 1.0) <= tol(len(h)))
    assert abs(got["iters"] - len(h)) <= (1 if near else 0), (got["iters"], len(h))
    m = min(got["iters"], len(h))
    for k in range(m):
        assert abs(got["hist"][k] - h[k]) <= tol(k) * h[k], (k, got["hist"][k], h[k])
    if got["iters"] == len(h):
        assert np.max(np.abs(got["x"] - x)) <= tol(m) * np.max(np.abs(x))
    again = run_cg(rowp, indx, vals, b, stop, 200, engine=mxm.CG_GRAPH)
    assert np.array_equal(got["x"], again["x"]) and got["r2"] == again["r2"]


@pytest.mark.parametrize("case", list(NEIGHBOURS))
def test_long_rows_beside_each_other(case):
    n, sets = NEIGHBOURS[case]
    rowp, indx, vals = coupled(n, sets(n))
    check(rowp, indx, vals, int(np.diff(rowp).max()))


@pytest.mark.parametrize("n,step,size", [(200000, 10, 600), (160000, 1600, 100), (8000, 16, 500)])
def test_long_rows_among_short_ones(n, step, size):
    """Every `step`-th row is coupled with `size - 1` others of its kind."""
    ids = np.arange(0, n, step)
    sets = [ids[i:i + size] for i in range(0, min(len(ids), 10 * size), size)]
    rowp, indx, vals = coupled(n, sets)
    check(rowp, indx, vals, int(np.diff(rowp).max()))


@pytest.mark.parametrize("n,full", [(160001, (0,)), (160001, (80000,)), (200000, (199999, 17, 18)),
                                    (40000, (0, 39999)), (17000, (3, 5, 7))])
def test_bordered(n, full):
    """A diagonal matrix with a few full rows and columns."""
    rng = np.random.default_rng(n)
    full = np.sort(np.asarray(full))
    rest = np.setdiff1d(np.arange(n), full)
    w = rng.uniform(-1, 1, (len(full), n)) / n
    length = np.full(n, len(full) + 1, dtype=np.int64)
    length[full] = n
    rowp = np.concatenate(([0], np.cumsum(length)))
    indx = np.empty(rowp[-1], dtype=np.int64)
    vals = np.empty(rowp[-1])
    for k, i in enumerate(full):
        indx[rowp[i]:rowp[i + 1]] = np.arange(n)
        row = w[k].copy()
        row[full] = (w[k][full] + w[:, i]) / 2  # symmetric where two full rows meet
        row[i] = 4.0
        vals[rowp[i]:rowp[i + 1]] = row
    cols = np.concatenate((np.broadcast_to(full, (len(rest), len(full))), rest[:, None]), axis=1)
    part = np.concatenate((w[:, rest].T, 2.0 + rng.uniform(0, 1, (len(rest), 1))), axis=1)
    o = np.argsort(cols, axis=1)
    at = rowp[rest][:, None] + np.arange(len(full) + 1)
    indx[at] = np.take_along_axis(cols, o, axis=1)
    vals[at] = np.take_along_axis(part, o, axis=1)
    check(rowp.astype(np.int32), indx.astype(np.int32), vals, n)


def test_wrong_pointers_and_columns():
    """Row pointers out of order, or columns outside, in a matrix with long rows
    are skipped and recorded."""
    n = 160001
    rowp, indx, vals = coupled(n, [np.arange(50, 700)])
    b = np.ones(n)
    for where, value in ((60, -5), (60, 2 ** 31 - 1), (300, 0), (n - 1, int(rowp[-1]) + 1)):
        bad = rowp.copy()
        bad[where] = value
        run_cg(bad, indx, vals, b, 0.0, 3, expect=mxm.MXM_ERR_INVALID_ARG, engine=mxm.CG_GRAPH)
    bad = indx.copy()
    bad[rowp[100] + 200] = n
    run_cg(rowp, bad, vals, b, 0.0, 3, expect=mxm.MXM_ERR_INVALID_ARG, engine=mxm.CG_GRAPH)


def test_one_row_of_twenty_million_values():
    """One block's product of such a row is not taken for a block that is lost:
    the step ends without MXM_ERR_TIMEOUT and its iterate is alpha b."""
    n = 20_000_000
    w = 0.1 / n
    rowp = torch.cat((torch.zeros(1, dtype=torch.int64),
                      n + 2 * torch.arange(n, dtype=torch.int64))).to(torch.int32).cuda()
    indx = torch.empty(3 * n - 2, dtype=torch.int32, device="cuda")
    vals = torch.empty(3 * n - 2, dtype=torch.float64, device="cuda")
    indx[:n] = torch.arange(n, dtype=torch.int32, device="cuda")
    vals[:n] = w
    vals[0] = 4.0
    indx[n::2] = 0
    indx[n + 1::2] = torch.arange(1, n, dtype=torch.int32, device="cuda")
    vals[n::2] = w
    vals[n + 1::2] = 2.0
    b = torch.ones(n, dtype=torch.float64, device="cuda")
    x = torch.empty_like(b)
    it, _ = mxm.mxm_cg(vals, indx, rowp, b, x, 0.0, 1, engine=mxm.CG_GRAPH)
    assert mxm.mxm_get_device_status() == mxm.MXM_OK and int(it) == 1
    # b = 1: (b, b) = n, (b, A b) = 4 + 2 (n - 1) + 2 w (n - 1)
    alpha = n / (4 + 2 * (n - 1) + 2 * w * (n - 1))
    assert float((x - alpha).abs().max()) <= 4 * n * U * alpha
