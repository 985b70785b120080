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


@pytest.mark.parametrize("precond", [0, 2])
@pytest.mark.parametrize("prec_name", ["FP64", "FP32_REFINE"])
@pytest.mark.parametrize("sizes", [
    [300, 512, 257, 31, 512],                    # no level below the finest
    [513, 20000, 300, 4097, 32, 9000, 256, 700],  # levels that some of the requests lack
], ids=["one-level", "uneven"])
def test_requests_that_finish_at_different_times_equal_those_alone(sizes, prec_name, precond):
    """The blocks of a batch share out the running requests' units, again whenever
    one finishes; every request's bits are those of the request alone."""
    dev = cuda_or_skip()
    from paper_1603_04100_gb300 import api
    from paper_1603_04100_gb300.batch import BatchPipeline
    prec = getattr(api, prec_name)
    clouds = [I.random_sphere(n, 70 + i) if i % 2 else I.torus(n, 70 + i) for i, n in enumerate(sizes)]
    cols = [1 + i % 3 for i in range(len(sizes))]
    fs = [p[:, :c] * (1.0 + p[:, 1:2]) for p, c in zip(clouds, cols)]
    spec = [(len(p), 12, c) for p, c in zip(clouds, cols)]
    dp = [torch.from_numpy(np.ascontiguousarray(p)).to(dev) for p in clouds]
    df = [torch.from_numpy(np.ascontiguousarray(f)).to(dev) for f in fs]
    both = BatchPipeline(spec, prec=prec, precond=precond, device=dev, rtol=1e-9)
    both.run(dp, df)
    torch.cuda.synchronize()
    its = set()
    for i, s in enumerate(spec):
        solo = BatchPipeline([s], prec=prec, precond=precond, device=dev, rtol=1e-9)
        solo.run([dp[i]], [df[i]])
        torch.cuda.synchronize()
        assert torch.equal(solo.slots[0].u, both.slots[i].u), (i, s)
        its.update(info[0] for info in both.infos()[i])
    # they did finish at different times (with one level the V-cycle is a direct solve)
    assert len(its) > 1 or (precond == 2 and max(sizes) <= 512)


def test_more_requests_than_the_list_holds():
    """700 small requests in one launch: past the list's room the runs are cut from
    all requests' units; the same bits as alone."""
    dev = cuda_or_skip()
    from paper_1603_04100_gb300 import api
    from paper_1603_04100_gb300.batch import BatchPipeline
    n, count = 96, 700
    clouds = [torch.from_numpy(I.random_sphere(n + i % 7, i)).to(dev) for i in range(count)]
    fs = [p[:, :1].clone() for p in clouds]
    spec = [(len(p), 8, 1) for p in clouds]
    both = BatchPipeline(spec, prec=api.FP32_REFINE, precond=2, device=dev, rtol=1e-9)
    both.run(clouds, fs)
    torch.cuda.synchronize()
    assert all(info[0][3] == 0 for info in both.infos())
    for i in (0, 1, 350, 698, 699):
        solo = BatchPipeline(spec[i:i + 1], prec=api.FP32_REFINE, precond=2, device=dev, rtol=1e-9)
        solo.run(clouds[i:i + 1], fs[i:i + 1])
        torch.cuda.synchronize()
        assert torch.equal(solo.slots[0].u, both.slots[i].u), i
