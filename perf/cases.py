"""Workloads of the library as its users run them, each through the public
entry points of ``paper_1211_1581_gb300.mxm``: the dense product (native
FP64 and the three bf16-digit splits), the grouped product, the sparse
product, conjugate gradients and the FFT.  Shapes are those of the
repository's benchmark suite and tests, from single small calls, where
launches and latency count, to the largest products."""
import math

import torch

from paper_1211_1581_gb300 import mxm

MODES = {"f64": mxm.MODE_F64, "i8": mxm.MODE_EMUL_I8, "bf16": mxm.MODE_EMUL_BF16,
         "rn8": mxm.MODE_EMUL_RN8}


def _gemm(name, mode, m, k, n, slices, values):
    return {"name": name, "op": "gemm", "mode": mode, "m": m, "k": k, "n": n, "slices": slices,
            "values": values}


def listed():
    return [
        # one small product: a call inside somebody's loop, launch-bound
        _gemm("f64_256", "f64", 256, 256, 256, 0, "uniform"),
        # the middle of the native FP64 sweep
        _gemm("f64_2048", "f64", 2048, 2048, 2048, 0, "uniform"),
        # a mid-size product whose dimensions fit no tile, 8-bit digits
        _gemm("bf16_1000x1777x1300", "bf16", 1000, 1777, 1300, 6, "spread"),
        # the headline product: FP64-accurate 8192^3 of widely spread entries
        _gemm("i8_8192", "i8", 8192, 8192, 8192, 7, "spread"),
        # the three rectangular products: a rank-256 update of a large C, an
        # inner product of long panels, a tall-skinny panel times a block
        _gemm("i8_16384x256x16384", "i8", 16384, 256, 16384, 6, "uniform"),
        _gemm("i8_128x65536x128", "i8", 128, 65536, 128, 6, "uniform"),
        _gemm("rn8_32768x1024x64", "rn8", 32768, 1024, 64, 6, "uniform"),
        # thousands of uneven small products in one grouped call
        {"name": "grouped_i8_2000", "op": "grouped", "mode": "i8", "count": 2000, "slices": 8,
         "sizes": 0},
        # a sparse matrix larger than L2, short rows
        {"name": "spmv_2m_mean16", "op": "spmv", "rows": 2000000, "cols": 2000000, "mean": 16.0},
        # a solve of the paper's Table 2 size, latency-bound, and a large one
        {"name": "cg_1024_bw127", "op": "cg", "n": 1024, "bw": 127},
        {"name": "cg_1m_bw7", "op": "cg", "n": 1000000, "bw": 7},
        # a transform of 2^20 points
        {"name": "fft_1m", "op": "fft", "log2n": 20},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["f64", "emul", "emul", "emul", "grouped", "spmv", "cg", "fft"])
    if op == "f64":
        m, k, n = (_log_int(rng, 64, 2048) for _ in range(3))
        return {"op": "gemm", "mode": "f64", "m": m, "k": k, "n": n, "slices": 0,
                "values": "uniform"}
    if op == "emul":
        mode = rng.choice(["i8", "i8", "bf16", "rn8"])
        values = rng.choice(["uniform", "spread"])
        m, k, n = (_log_int(rng, 64, 8192) for _ in range(3))
        slices = (6 if values == "uniform" else 7) + (mode == "i8") - 1
        return {"op": "gemm", "mode": mode, "m": m, "k": k, "n": n, "slices": slices,
                "values": values}
    if op == "grouped":
        mode = rng.choice(["f64", "i8", "rn8"])
        return {"op": "grouped", "mode": mode, "count": _log_int(rng, 100, 1500),
                "slices": {"f64": 0, "i8": 8, "rn8": 7}[mode], "sizes": rng.randrange(1, 1000)}
    if op == "spmv":
        rows = _log_int(rng, 1000, 1500000)
        mean = round(math.exp(rng.uniform(math.log(4), math.log(min(256.0, 3e7 / rows)))), 1)
        return {"op": "spmv", "rows": rows, "cols": max(1024, rows + rng.randrange(-500, 500)),
                "mean": mean}
    if op == "cg":
        n = _log_int(rng, 128, 800000)
        half = _log_int(rng, 1, min(255, n // 4, max(1, 4000000 // n)))
        return {"op": "cg", "n": n, "bw": 2 * half + 1}
    return {"op": "fft", "log2n": rng.randrange(4, 22)}


def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _values(kind, shape, g):
    """Entries uniform in [-1, 1), or s u 2^e: random sign, u in [1, 2), e an
    integer in [-20, 20]."""
    x = torch.rand(shape, dtype=torch.float64, device="cuda", generator=g)
    if kind == "uniform":
        return x.mul_(2.0).sub_(1.0)
    e = torch.randint(-20, 21, shape, device="cuda", generator=g, dtype=torch.int32)
    x = torch.ldexp(x.add_(1.0), e)
    s = torch.randint(0, 2, shape, device="cuda", generator=g, dtype=torch.int8)
    return x.mul_(s.mul_(2).sub_(1))


def _gemm_inputs(case, seed):
    g = _generator(seed)
    return (_values(case["values"], (case["m"], case["k"]), g),
            _values(case["values"], (case["k"], case["n"]), g))


def _grouped_dims(case):
    """(m, k, n) of each problem, every dimension log-uniform in [16, 1024]:
    the batch's sizes belong to the case, its values to the seed."""
    g = torch.Generator()
    g.manual_seed(case["sizes"])
    u = torch.rand((case["count"], 3), dtype=torch.float64, generator=g)
    v = torch.exp(math.log(16.0) + u * math.log(64.0)).round().clamp(16, 1024)
    return v.to(torch.int64).tolist()


def _grouped_inputs(case, seed):
    """The problems' operands, packed one after another in two buffers."""
    dims = _grouped_dims(case)
    g = _generator(seed)
    a = _values("uniform", (sum(m * k for m, k, _ in dims),), g)
    b = _values("uniform", (sum(k * n for _, k, n in dims),), g)
    views, oa, ob = [], 0, 0
    for m, k, n in dims:
        views.append((a[oa:oa + m * k].view(m, k), b[ob:ob + k * n].view(k, n)))
        oa += m * k
        ob += k * n
    return dims, views


def _csr_inputs(case, seed):
    """Rows of near-binomial length around the mean, columns uniform and
    increasing within a row, values uniform in [-1, 1)."""
    rows, cols, mean = case["rows"], case["cols"], case["mean"]
    g = _generator(seed)
    z = torch.randn(rows, dtype=torch.float64, device="cuda", generator=g)
    want = (mean + math.sqrt(mean) * z).round().clamp(0, min(cols, 4 * mean + 16)).to(torch.int64)
    row = torch.repeat_interleave(torch.arange(rows, device="cuda"), want)
    col = torch.randint(0, cols, (row.numel(),), device="cuda", generator=g)
    key = torch.unique(row * cols + col)
    row = torch.div(key, cols, rounding_mode="floor")
    rowp = torch.zeros(rows + 1, dtype=torch.int64, device="cuda")
    rowp[1:] = torch.cumsum(torch.bincount(row, minlength=rows), 0)
    indx = (key - row * cols).to(torch.int32)
    vals = _values("uniform", (key.numel(),), g)
    x = _values("uniform", (cols,), g)
    return vals, indx, rowp.to(torch.int32), x


def _cg_inputs(case, seed):
    """A random symmetric, strictly diagonally dominant band matrix in CSR
    and a right-hand side (the solver's Table 2 kind of system)."""
    n, h = case["n"], (case["bw"] - 1) // 2
    g = _generator(seed)
    up = _values("uniform", (n, h), g)
    band = torch.zeros((n, 2 * h + 1), dtype=torch.float64, device="cuda")
    for d in range(1, h + 1):
        band[:n - d, h + d] = up[:n - d, d - 1]
        band[d:, h - d] = up[:n - d, d - 1]
    band[:, h] = 1.0 + band.abs().sum(dim=1)
    cols = (torch.arange(n, device="cuda")[:, None]
            + torch.arange(-h, h + 1, device="cuda")[None, :])
    keep = (cols >= 0) & (cols < n)
    rowp = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    rowp[1:] = torch.cumsum(keep.sum(dim=1), 0)
    b = _values("uniform", (n,), g)
    return band[keep], cols[keep].to(torch.int32), rowp.to(torch.int32), b


def _fft_input(case, seed):
    g = _generator(seed)
    return torch.view_as_complex(_values("uniform", (1 << case["log2n"], 2), g))


def prepare(case, seed):
    state = {"case": case}
    if case["op"] == "gemm":
        A, B = _gemm_inputs(case, seed)
        C = torch.empty((case["m"], case["n"]), dtype=torch.float64, device="cuda")
        state.update(A=A, B=B, C=C)
    elif case["op"] == "grouped":
        dims, views = _grouped_inputs(case, seed)
        c = torch.empty(sum(m * n for m, _, n in dims), dtype=torch.float64, device="cuda")
        problems, oc = [], 0
        for (m, _, n), (A, B) in zip(dims, views):
            problems.append((A, B, c[oc:oc + m * n].view(m, n)))
            oc += m * n
        table = mxm.problem_table(problems)
        need = mxm.mxm_grouped_workspace_size(table, MODES[case["mode"]], case["slices"])
        ws = torch.empty(max(1, need), dtype=torch.uint8, device="cuda")
        state.update(problems=problems, table=table.cuda(), ws=ws, C=c)
    elif case["op"] == "spmv":
        vals, indx, rowp, x = _csr_inputs(case, seed)
        y = torch.empty(case["rows"], dtype=torch.float64, device="cuda")
        state.update(vals=vals, indx=indx, rowp=rowp, x=x, y=y)
    elif case["op"] == "cg":
        vals, indx, rowp, b = _cg_inputs(case, seed)
        n = case["n"]
        work = torch.empty((mxm.load().mxm_cg_workspace_size(n) + 7) // 8, dtype=torch.float64,
                           device="cuda")
        state.update(vals=vals, indx=indx, rowp=rowp, b=b, work=work,
                     x=torch.empty(n, dtype=torch.float64, device="cuda"),
                     iters=torch.zeros(1, dtype=torch.int32, device="cuda"),
                     r2=torch.zeros(1, dtype=torch.float64, device="cuda"),
                     stop=1e-24 * float(b @ b))
    else:
        x = _fft_input(case, seed)
        state.update(x=x, out=torch.empty_like(x), fft=mxm.FFT(1 << case["log2n"]))
    return state


def run(state):
    case = state["case"]
    if case["op"] == "gemm":
        if case["mode"] == "f64":
            return mxm.mxm_f64(state["A"], state["B"], state["C"])
        return mxm.mxm_gemm(MODES[case["mode"]], state["A"], state["B"], state["C"],
                            case["slices"])
    if case["op"] == "grouped":
        mxm.mxm_grouped(state["table"], MODES[case["mode"]], case["slices"], state["ws"])
        return state["C"]
    if case["op"] == "spmv":
        return mxm.mxm_spmv(state["vals"], state["indx"], state["rowp"], state["x"], state["y"])
    if case["op"] == "cg":
        iters, r2 = mxm.mxm_cg(state["vals"], state["indx"], state["rowp"], state["b"],
                               state["x"], state["stop"], 1000, iters=state["iters"],
                               r2=state["r2"], work=state["work"])
        return {"x": state["x"], "iters": iters, "r2": r2}
    return state["fft"](state["x"], out=state["out"])


def work(case):
    """Bytes: each input read once, each output written once.  Flops: the
    FP64 operations of the definition (2 m k n of a product, whatever the
    engine computes it with; one step of the solver, whose step count is
    the data's; 5 n log2 n of the transform)."""
    if case["op"] == "gemm":
        m, k, n = case["m"], case["k"], case["n"]
        return {"bytes": 8 * (m * k + k * n + m * n), "flops": 2 * m * k * n}
    if case["op"] == "grouped":
        dims = _grouped_dims(case)
        return {"bytes": 8 * sum(m * k + k * n + m * n for m, k, n in dims),
                "flops": 2 * sum(m * k * n for m, k, n in dims)}
    if case["op"] == "spmv":
        nnz = case["rows"] * case["mean"]
        return {"bytes": 12 * nnz + 12 * case["rows"] + 8 * case["cols"], "flops": 2 * nnz}
    if case["op"] == "cg":
        nnz = case["n"] * case["bw"]
        return {"bytes": 12 * nnz + 20 * case["n"], "flops": 2 * nnz + 10 * case["n"]}
    n = 1 << case["log2n"]
    return {"bytes": 32 * n, "flops": 5 * n * case["log2n"]}


def exact(case, seed):
    if case["op"] == "gemm":
        A, B = _gemm_inputs(case, seed)
        return A @ B
    if case["op"] == "grouped":
        return torch.cat([(A @ B).reshape(-1) for A, B in _grouped_inputs(case, seed)[1]])
    if case["op"] == "spmv":
        vals, indx, rowp, x = _csr_inputs(case, seed)
        row = torch.repeat_interleave(torch.arange(case["rows"], device="cuda"),
                                      rowp.diff().to(torch.int64))
        y = torch.zeros(case["rows"], dtype=torch.float64, device="cuda")
        return y.index_add_(0, row, vals * x[indx.to(torch.int64)])
    if case["op"] == "cg":
        # the solution itself: the same iteration carried on to the rounding
        vals, indx, rowp, b = _cg_inputs(case, seed)
        row = torch.repeat_interleave(torch.arange(case["n"], device="cuda"),
                                      rowp.diff().to(torch.int64))
        col = indx.to(torch.int64)
        x, r, p = torch.zeros_like(b), b.clone(), b.clone()
        r2 = float(r @ r)
        stop = 1e-30 * r2
        for _ in range(300):
            if r2 <= stop:
                break
            q = torch.zeros_like(b).index_add_(0, row, vals * p[col])
            alpha = r2 / float(p @ q)
            x.add_(p, alpha=alpha)
            r.sub_(q, alpha=alpha)
            r2, old = float(r @ r), r2
            p.mul_(r2 / old).add_(r)
        return {"x": x, "iters": None, "r2": None}
    return torch.fft.fft(_fft_input(case, seed))
