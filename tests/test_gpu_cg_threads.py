"""Conjugate gradients over all SMs from two host threads at once, on a stream
each, with systems whose blocks use very different amounts of shared memory:
every solve is accepted and gives the bits of the same solve alone."""
import threading

import numpy as np
import pytest

from paper_1211_1581_gb300 import inputs

torch = pytest.importorskip("torch")
from paper_1211_1581_gb300 import mxm  # noqa: E402

pytestmark = pytest.mark.gpu


class System:
    def __init__(self, seed, n, bw):
        rowp, indx, vals = inputs.banded_spd(seed, 122, n, bw)
        self.a = [torch.from_numpy(np.ascontiguousarray(v)).cuda() for v in (vals, indx, rowp)]
        self.b = torch.from_numpy(inputs.uniform_pm1(seed, 123, (n,))).cuda()
        self.x = torch.empty(n, dtype=torch.float64, device="cuda")
        self.work = torch.empty((mxm.load().mxm_cg_workspace_size(n) + 7) // 8,
                                dtype=torch.float64, device="cuda")
        self.it = torch.zeros(1, dtype=torch.int32, device="cuda")
        self.r2 = torch.zeros(1, dtype=torch.float64, device="cuda")

    def solve(self, steps, stream=None):
        mxm.mxm_cg(*self.a, self.b, self.x, 0.0, steps, self.it, self.r2, engine=mxm.CG_GRAPH,
                   work=self.work, stream=stream)


@pytest.mark.parametrize("sizes", [((160000, 5), (900000, 3)), ((1500000, 3), (900000, 3)),
                                   ((200, 3), (4000, 3))])
def test_two_threads(sizes):
    systems = [System(40 + i, *s) for i, s in enumerate(sizes)]  # one lane count for both
    want = []
    for s in systems:
        s.solve(3)
        torch.cuda.synchronize()
        want.append(s.x.clone())
    refused = []
    start = threading.Barrier(2)

    def go(s):
        stream = torch.cuda.Stream()
        start.wait()
        for _ in range(1500):
            try:
                s.solve(0, stream)
            except mxm.MxmError as e:
                refused.append(e.status)
        s.solve(3, stream)

    threads = [threading.Thread(target=go, args=(s,)) for s in systems]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert refused == []
    assert mxm.mxm_get_device_status() == mxm.MXM_OK
    for s, w in zip(systems, want):
        assert torch.equal(s.x, w)
