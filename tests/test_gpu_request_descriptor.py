"""A request descriptor whose number of right-hand sides is not the request's: the
launch sizes its registers, states and groups by the descriptor, so it does no work and
reports MVGD_EINVAL; the same request then solves with the right descriptor."""
from __future__ import annotations

import numpy as np
import pytest

from paper_1603_04100_gb300 import inputs as I
from tests.gpu_util import cuda_or_skip

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precond", [0, 2])
@pytest.mark.parametrize("prec_name", ["FP64", "FP32_REFINE"])
@pytest.mark.parametrize("nrhs,said", [(3, 8), (4, 6), (3, 1), (8, 2), (1, 4), (5, 4)])
def test_wrong_number_of_right_hand_sides_is_refused(nrhs, said, prec_name, precond):
    dev = cuda_or_skip()
    from paper_1603_04100_gb300 import _lib as LB
    from paper_1603_04100_gb300 import api
    from paper_1603_04100_gb300.batch import BatchPipeline
    prec = getattr(api, prec_name)
    p = I.random_sphere(1500, 95)
    x, y, z = p.T
    f = np.stack([x, y * z, z, x * y, 5 * z ** 3 - 3 * z, np.sin(x), x * x - y * y, 1 + x * z][:nrhs], axis=1)
    pts, fs = [torch.from_numpy(p).to(dev)], [torch.from_numpy(np.ascontiguousarray(f)).to(dev)]
    pipe = BatchPipeline([(1500, 20, nrhs)], prec=prec, precond=precond, device=dev, rtol=1e-9)
    right, slot, L = pipe._reqs, pipe.slots[0], LB.load()
    pipe._reqs = LB.requests([(slot.req_ws, slot.n, said, slot.k)])
    pipe.run(pts, fs)  # initialised for nrhs, listed with `said`
    torch.cuda.synchronize()
    info = pipe.infos()[0]
    if said > nrhs and all(i[3] == 0 for i in info):
        pass  # wider than needed and not cut into groups: solved
    else:
        assert [(i[0], i[3]) for i in info] == [(0, LB.EINVAL)] * nrhs
        LB.check("mvgd_iterate", L.mvgd_iterate(right, 1, prec, precond, pipe.budget, None, api._vp(pipe.ctl_ws),
                                                 pipe.ctl_ws.numel(), api._stream()))
        LB.check("mvgd_request_finish", L.mvgd_request_finish(api._vp(slot.req_ws), slot.n, nrhs, api._vp(slot.u),
                                                               api._vp(slot.info), api._stream()))
        torch.cuda.synchronize()
    through = BatchPipeline([(1500, 20, nrhs)], prec=prec, precond=precond, device=dev, rtol=1e-9)
    through.run(pts, fs)
    torch.cuda.synchronize()
    assert pipe.infos() == through.infos() and torch.equal(slot.u, through.slots[0].u)
