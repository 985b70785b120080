"""Two staged slices a warp selected, for launches of several requests (which keep to
one) and of one large request: the bits are those of one slice a warp."""
from __future__ import annotations

import numpy as np
import pytest

from paper_1603_04100_gb300 import inputs as I
from tests.gpu_util import cuda_or_skip

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precond", [1, 2])
@pytest.mark.parametrize("prec_name", ["FP64", "FP32_REFINE"])
@pytest.mark.parametrize("sizes", [[3000, 3000], [513, 90000, 300, 4097, 32, 9000, 256, 700], [200000]],
                         ids=["two", "uneven", "one"])
def test_two_slices_a_warp_give_the_same_bits(sizes, prec_name, precond):
    dev = cuda_or_skip()
    from paper_1603_04100_gb300 import api
    from paper_1603_04100_gb300 import tune
    from paper_1603_04100_gb300.batch import BatchPipeline
    if precond == 1 and max(sizes) > 5000:
        pytest.skip("the row-scaled flows take the same dispatch at the small sizes")
    clouds = [I.random_sphere(n, 100 + i) for i, n in enumerate(sizes)]
    spec = [(n, 12 if n == 32 else 20, 1 + i % 3) for i, n in enumerate(sizes)]
    pts = [torch.from_numpy(p).to(dev) for p in clouds]
    fs = [torch.from_numpy(np.ascontiguousarray(p[:, :q] * (1.0 + p[:, 1:2]))).to(dev)
          for p, (_, _, q) in zip(clouds, spec)]
    got = []
    try:
        for buffers in (1, 2):
            tune.Tuning(stage_buffers=buffers).apply()
            b = BatchPipeline(spec, prec=getattr(api, prec_name), precond=precond, device=dev, rtol=1e-9)
            b.run(pts, fs)
            torch.cuda.synchronize()
            got.append((b.infos(), [s.u.clone() for s in b.slots]))
    finally:
        tune.Tuning().apply()
    assert got[0][0] == got[1][0]
    assert all(torch.equal(a, b) for a, b in zip(got[0][1], got[1][1]))
