"""Calls of different sizes from several host threads, each on its own stream: a launch
needs the shared memory of its own size, whatever another thread has just launched."""
from __future__ import annotations

import threading

import numpy as np
import pytest

from paper_1603_04100_gb300 import inputs as I
from tests.gpu_util import cuda_or_skip

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec_name", ["FP64", "FP32_REFINE"])
def test_threads_of_different_sizes(prec_name):
    dev = cuda_or_skip()
    from paper_1603_04100_gb300 import api
    prec = getattr(api, prec_name)
    work = []
    for n, k in ((200, 8), (512, 31), (129, 12), (400, 24)):
        p = torch.from_numpy(I.random_sphere(n, n)).to(dev)
        nbr = api.knn(p, k)
        op = api.assemble(p, nbr, prec=prec)
        want = (op.weights(), api.amg_setup(op).coarsest_inverse())
        work.append((p, nbr, k, want))
    torch.cuda.synchronize()
    errors = []

    def calls(p, nbr, k, want):
        try:
            s = torch.cuda.Stream(device=dev)
            with torch.cuda.stream(s):
                for i in range(400):
                    op = api.assemble(p, nbr, prec=prec)
                    H = api.amg_setup(op)
                s.synchronize()
                assert np.array_equal(op.weights(), want[0]) and np.array_equal(H.coarsest_inverse(), want[1])
        except Exception as e:  # noqa: BLE001
            errors.append(repr(e))

    threads = [threading.Thread(target=calls, args=w) for w in work]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
