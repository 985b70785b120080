"""kNN at the limits of its input: extents that are not finite, clouds so small or large
that FP32 squares of their distances are not normal numbers, and points far denser
than the search grid."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
from paper_1603_04100_gb300 import inputs as I
from tests.gpu_util import cuda_or_skip

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _spoilt(kind):
    p = I.random_sphere(3000, 30)
    axis = {"x": 0, "y": 1, "z": 2}[kind[0]]
    if kind[1:] == "+inf":
        p[17, axis] = np.inf
    elif kind[1:] == "-inf":
        p[17, axis] = -np.inf
    elif kind[1:] == "inf both":
        p[17, axis], p[2040, axis] = np.inf, -np.inf
    elif kind[1:] == "overflow":  # finite points, an extent beyond FP64
        p[17, axis], p[2040, axis] = 1.7e308, -1.7e308
    else:
        p[:, axis] = np.nan
    return p


@pytest.mark.parametrize("kind", [a + b for a in "xyz" for b in ("+inf", "-inf", "inf both", "overflow", "nan")])
def test_extent_that_is_not_finite_gives_empty_lists(kind):
    """No cell grid exists: the lists come back empty, the rows as not finite, and the
    next cloud's lists are right."""
    dev = cuda_or_skip()
    from paper_1603_04100_gb300 import api
    pt = torch.from_numpy(_spoilt(kind)).to(dev)
    nbr, order = api.knn(pt, 20, want_order=True)
    assert bool((nbr == -1).all())
    assert torch.equal(torch.sort(order).values, torch.arange(len(pt), dtype=torch.int32, device=dev))
    for prec in (api.FP64, api.FP32_REFINE):
        op = api.assemble(pt, nbr, prec=prec, order=order)
        assert int(op.bad_rows.item()) == len(pt) and bool((op.status == 2).all())
    good = torch.from_numpy(I.random_sphere(3000, 30)).to(dev)
    assert int(api.knn(good, 20).min()) >= 0


@pytest.mark.parametrize("value", [np.nan, np.inf])
def test_a_few_points_that_are_not_numbers_leave_the_others_exact(value):
    """NaN coordinates are outside the box (an infinite one empties every list): the
    other points' lists are those of the cloud without them."""
    dev = cuda_or_skip()
    from paper_1603_04100_gb300 import api
    p = I.random_sphere(3000, 31)
    bad = np.array([5, 1200, 2999])
    q = p.copy()
    q[bad] = value
    nbr = api.knn(torch.from_numpy(q).to(dev), 12).cpu().numpy()
    if np.isinf(value):
        assert (nbr == -1).all()
        return
    keep = np.setdiff1d(np.arange(3000), bad)
    want = api.knn(torch.from_numpy(np.ascontiguousarray(p[keep])).to(dev), 12).cpu().numpy()
    np.testing.assert_array_equal(nbr[keep], keep[want])


@pytest.mark.parametrize("k", [6, 20, 31])
@pytest.mark.parametrize("scale", [1e-16, 1e-18, 1e-19, 3e-20, 1e-20, 3e-21, 1e-21, 1e-22, 1e-24, 1e-35, 1e15, 1e19, 1e25])
def test_lists_are_exact_where_fp32_squares_underflow_or_overflow(scale, k):
    """Squared distances that are subnormal (or zero, or infinite) in FP32: the screen's
    bound has to know their absolute error."""
    dev = cuda_or_skip()
    from paper_1603_04100_gb300 import api
    p = scale * I.random_sphere(2500, 32)
    nbr = api.knn(torch.from_numpy(p).to(dev), k).cpu().numpy()
    np.testing.assert_array_equal(nbr, oracle.knn_brute(p, k))


def _graded(n, seed):  # a sphere whose points crowd at two poles
    p = I.random_sphere(n, seed)
    z = np.sign(p[:, 2]) * (1 - (1 - np.abs(p[:, 2])) ** 3)
    rho = np.sqrt(np.maximum(1 - z * z, 0)) / np.hypot(p[:, 0], p[:, 1])
    return np.ascontiguousarray(np.stack([p[:, 0] * rho, p[:, 1] * rho, z], 1))


@pytest.mark.parametrize("k", [1, 20, 31])
@pytest.mark.parametrize("cell", [0.0, -2.0, 0.06, 0.4])
def test_queries_with_more_candidates_than_a_warp_holds(cell, k):
    """From a few hundred candidates in a query's cells to thousands inside its guard,
    ties and points that are not numbers among them."""
    dev = cuda_or_skip()
    from paper_1603_04100_gb300 import api
    p = _graded(6000, 33)
    p[100:140] = p[99]
    nbr = api.knn(torch.from_numpy(p).to(dev), k, cell_size=cell).cpu().numpy()
    np.testing.assert_array_equal(nbr, oracle.knn_brute(p, k))
    q = np.concatenate([p, np.full((50, 3), np.nan)])
    nbr = api.knn(torch.from_numpy(q).to(dev), k, cell_size=cell).cpu().numpy()
    np.testing.assert_array_equal(nbr[:6000], oracle.knn_brute(p, k))
