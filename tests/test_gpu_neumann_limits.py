"""A cloud without neighbour lists (an infinite coordinate) gives no ghosts: every boundary
frame is bad and the operator is refused."""
from __future__ import annotations

import numpy as np
import pytest

from paper_1603_04100_gb300 import inputs as I
from tests.gpu_util import cuda_or_skip

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_cloud_without_lists_is_refused():
    dev = cuda_or_skip()
    from paper_1603_04100_gb300 import api
    p, flags = I.hemisphere(3000, 5)
    boundary = torch.from_numpy(np.ascontiguousarray(flags).astype(np.uint8)).to(dev)
    good = torch.from_numpy(np.ascontiguousarray(p)).to(dev)
    bad = good.clone()
    bad[1500, 2] = float("inf")
    nbr = api.knn(bad, 20)
    assert bool((nbr == -1).all())
    cloud = api.neumann_ghosts(bad, nbr, boundary)
    assert cloud.n_ghost == 0 and cloud.bad_frames == cloud.n_boundary > 0
    with pytest.raises(api.MvgdError):
        api.neumann_operator(bad, boundary, 20)
    op, cloud = api.neumann_operator(good, boundary, 20)
    assert cloud.bad_frames == 0 and cloud.n_ghost > 0
