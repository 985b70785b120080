"""A launch stopped by its cancel word leaves every request at an iteration's end: a
request stopped after each of its iterations, restarts among them, and taken up again
gives the bits, the iteration and the refinement counts of one that ran through.  All
forms of a launch: one request of few tiles (its states kept by every block), one of
many, right-hand sides in groups, several requests."""
from __future__ import annotations

import numpy as np
import pytest

from paper_1603_04100_gb300 import inputs as I
from tests.gpu_util import cuda_or_skip

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SIZES = {
    "one": [(2000, 16, 1)], "groups": [(1500, 16, 4)], "wide": [(30000, 16, 8)], "odd": [(3001, 20, 3)],
    "many tiles": [(140000, 20, 1)], "several": [(1500, 16, 2), (700, 16, 1), (5000, 16, 1)],
}


@pytest.mark.parametrize("precond", [0, 1, 2])
@pytest.mark.parametrize("prec_name", ["FP64", "FP32_REFINE"])
@pytest.mark.parametrize("case", list(SIZES))
def test_cancelled_request_resumes_where_it_stopped(case, prec_name, precond):
    dev = cuda_or_skip()
    from paper_1603_04100_gb300 import _lib as LB
    from paper_1603_04100_gb300 import api
    from paper_1603_04100_gb300.batch import BatchPipeline
    sizes = SIZES[case]
    if precond != 2 and sizes[0][0] > 5000:
        pytest.skip("the row-scaled flows take the same dispatch at the small sizes")
    prec = getattr(api, prec_name)
    clouds = [I.random_sphere(n, 80 + i) for i, (n, _, _) in enumerate(sizes)]
    fs = []
    for p, (_, _, q) in zip(clouds, sizes):
        x, y, z = p.T
        fs.append(np.stack([x, y * z, z, x * y, 5 * z ** 3 - 3 * z, np.sin(x), x * x - y * y, 1 + x * z][:q], axis=1))
    pts = [torch.from_numpy(p).to(dev) for p in clouds]
    f = [torch.from_numpy(np.ascontiguousarray(a)).to(dev) for a in fs]
    through = BatchPipeline(sizes, prec=prec, precond=precond, device=dev, rtol=1e-9)
    through.run(pts, f)
    torch.cuda.synchronize()
    want = through.infos()
    assert all(i[3] == 0 for s in want for i in s)
    L = LB.load()
    stop = torch.ones(1, dtype=torch.int32, device=dev)
    pipe = BatchPipeline(sizes, prec=prec, precond=precond, device=dev, rtol=1e-9)
    pipe.run(pts, f, cancel=stop)  # every request's first iteration (its first restart)
    torch.cuda.synchronize()
    assert any(i[3] == LB.ECANCELLED for s in pipe.infos() for i in s)
    for launch in range(2000):
        LB.check("mvgd_iterate", L.mvgd_iterate(pipe._reqs, len(pipe.slots), prec, precond, pipe.budget, api._vp(stop),
                                                 api._vp(pipe.ctl_ws), pipe.ctl_ws.numel(), api._stream()))
        if launch % 16 == 15:
            for s in pipe.slots:
                LB.check("mvgd_request_finish", L.mvgd_request_finish(api._vp(s.req_ws), s.n, s.nrhs, api._vp(s.u),
                                                                       api._vp(s.info), api._stream()))
            torch.cuda.synchronize()
            if all(i[3] == 0 for s in pipe.infos() for i in s):
                break
    assert pipe.infos() == want
    assert all(torch.equal(a.u, b.u) for a, b in zip(pipe.slots, through.slots))
