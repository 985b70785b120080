"""The coarsest level of a one-level hierarchy where a row names a column twice, or
itself, as the rows folded over a Neumann boundary do: each slot adds to the matrix,
as it does in the operator's products.  Bounds: a Gauss-Jordan inverse in FP32 and one
refined in FP64, 4 n u cond(A)."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
from paper_1603_04100_gb300 import inputs as I
from tests.gpu_util import cuda_or_skip, operator_from_rows

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec_name", ["FP64", "FP32_REFINE"])
@pytest.mark.parametrize("n", [9, 40, 65, 300, 512])
def test_repeated_columns_add_up(n, prec_name):
    dev = cuda_or_skip()
    from paper_1603_04100_gb300 import api
    k = 8
    pts = I.morton_sorted(I.random_sphere(n, 90))
    nbr = oracle.knn_grid(pts, k).copy()
    r = np.random.default_rng(91)
    val = np.zeros((n, k + 1))
    val[:, 1:] = r.uniform(0.5, 2.0, (n, k))
    val[:, 0] = -val[:, 1:].sum(1)
    nbr[::2, 3] = nbr[::2, 2]             # a column twice
    nbr[::5, 4] = nbr[::5, 2]             # and three times in some rows
    nbr[::3, 5] = np.arange(n)[::3]       # the row itself
    nbr[::6, 6] = np.arange(n)[::6]
    op = operator_from_rows(nbr, val, getattr(api, prec_name), dev)
    w = op.weights()                      # what is stored (hi + lo in the mixed format)
    A = np.zeros((n, n))
    np.add.at(A, (np.repeat(np.arange(n), k), nbr.ravel()), -w[:, 1:].ravel())
    A[np.arange(n), np.arange(n)] += 1.0 - w[:, 0]
    H = api.amg_setup(op, 1.0)
    assert H.levels == 1 and H.info(0).status == 0
    want, cond = np.linalg.inv(A), np.linalg.cond(A)
    for fp64, u in ((False, 2.0 ** -24), (True, 2.0 ** -53)):
        X = H.coarsest_inverse(fp64=fp64).astype(np.float64)
        assert np.linalg.norm(X - want) / np.linalg.norm(want) <= 4 * n * u * cond
    # the V-cycle of one level is this inverse: one or two iterations
    f = torch.from_numpy(np.stack([np.sin(pts[:, 0]), pts[:, 1]], 1).copy()).to(dev)
    res = api.solve(op, f, rtol=1e-10, precond=2, amg=H)
    assert res.status == [0, 0]
    err = np.linalg.norm(res.u.cpu().numpy() - want @ f.cpu().numpy()) / np.linalg.norm(want @ f.cpu().numpy())
    assert err <= 1e-10 * cond + 4 * n * 2.0 ** -53 * cond
