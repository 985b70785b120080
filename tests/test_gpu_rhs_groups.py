"""A request solved alone may have its right-hand sides cut into groups and its
level-0 tiles on other blocks than in a batch; each right-hand side's result must
not depend on either.  Every grouping of 2 .. 8 right-hand sides, both formats, all
preconditioners, against the same cloud inside a batch (where nothing is cut): the
same bits, and residuals at the tolerance."""
from __future__ import annotations

import numpy as np
import pytest

from paper_1603_04100_gb300 import inputs as I
from tests.gpu_util import cuda_or_skip

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precond", [0, 1, 2])
@pytest.mark.parametrize("prec_name", ["FP64", "FP32_REFINE"])
@pytest.mark.parametrize("n,nrhs", [(513, 2), (3001, 3), (3001, 8), (20000, 5), (20000, 6), (40001, 4)])
def test_right_hand_sides_alone_equal_those_in_a_batch(n, nrhs, prec_name, precond):
    dev = cuda_or_skip()
    from paper_1603_04100_gb300 import api
    from paper_1603_04100_gb300.batch import BatchPipeline
    if precond != 2 and n > 5000:
        pytest.skip("the row-scaled flows take the same dispatch at the small sizes")
    prec = getattr(api, prec_name)
    p, other = I.random_sphere(n, 60), I.torus(700, 61)
    x, y, z = p.T
    f = np.stack([x, y * z, z, x * y, 5 * z ** 3 - 3 * z, np.sin(x), x * x - y * y, 1 + x * z][:nrhs], axis=1).copy()
    pts = [torch.from_numpy(p).to(dev), torch.from_numpy(other).to(dev)]
    fs = [torch.from_numpy(f).to(dev), torch.from_numpy(other[:, :1].copy()).to(dev)]
    sizes = [(n, 16, nrhs), (700, 16, 1)]
    both = BatchPipeline(sizes, prec=prec, precond=precond, device=dev, rtol=1e-9)
    solo = BatchPipeline(sizes[:1], prec=prec, precond=precond, device=dev, rtol=1e-9)
    both.run(pts, fs)
    solo.run(pts[:1], fs[:1])
    torch.cuda.synchronize()
    assert torch.equal(solo.slots[0].u, both.slots[0].u)
    assert all(st == 0 and rel <= 1e-9 for _, _, rel, st in solo.infos()[0]), solo.infos()[0]
