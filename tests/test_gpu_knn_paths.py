"""kNN lists and the exported row order at the edges of the search's paths: the
screened query (few candidates), its exact re-rank (ties and near ties), the general
scan (too many candidates, rings beyond the first), wrapped and degenerate cell grids,
and both sorts of the row order with their switch.  Integer results: exact."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
from paper_1603_04100_gb300 import inputs as I
from tests.gpu_util import cuda_or_skip

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _rng(s):
    return np.random.default_rng(s)


def _lattice(m):  # every distance tied many times over
    g = np.stack(np.meshgrid(*[np.arange(m, dtype=np.float64)] * 3, indexing="ij"), -1).reshape(-1, 3)
    return np.ascontiguousarray(g[_rng(1).permutation(len(g))])


def _clusters():  # dense knots: thousands of candidates in a cell, sparse points between
    r = _rng(2)
    return np.concatenate([r.normal(c, 1e-4, (1500, 3)) for c in r.uniform(-1, 1, (4, 3))] + [r.uniform(-1, 1, (500, 3))])


def _duplicates():
    p = I.random_sphere(4000, 3)
    p[1000:1200] = p[999]
    p[2000:2040] = p[1999]
    return p


CLOUDS = {
    "sphere_8191": lambda: I.random_sphere(8191, 4), "sphere_8192": lambda: I.random_sphere(8192, 5),
    "sphere_8193": lambda: I.random_sphere(8193, 6), "torus_12289": lambda: I.torus(12289, 7),
    "lattice": lambda: _lattice(13), "clusters": _clusters, "duplicates": _duplicates,
    "line": lambda: np.stack([np.sort(_rng(8).uniform(0, 1, 3000)), np.zeros(3000), np.zeros(3000)], 1),
    "plane": lambda: np.concatenate([_rng(9).uniform(-1, 1, (5000, 2)), np.zeros((5000, 1))], 1),
    "far": lambda: I.random_sphere(3000, 10) + np.array([1e6, -2e5, 3e4]),
    "outlier": lambda: np.concatenate([I.random_sphere(3000, 11), [[1000.0, 1000.0, 1000.0]]]),
    "volume": lambda: _rng(12).uniform(0, 1, (9000, 3)),
    "tiny_scale": lambda: 1e-9 * I.ellipsoid(2500, 13),
}


def _order(pts):
    lo = pts.min(axis=0)
    e = float((pts.max(axis=0) - lo).max())
    q = np.clip((pts - lo) * (2097152.0 / e), 0.0, 2097151.0).astype(np.uint64)
    key = np.zeros(pts.shape[0], dtype=np.uint64)
    for b in range(21):
        for a in range(3):
            key |= ((q[:, a] >> np.uint64(b)) & np.uint64(1)) << np.uint64(3 * b + a)
    return np.lexsort((np.arange(len(pts)), key))


@pytest.mark.parametrize("k", [1, 5, 20, 31])
@pytest.mark.parametrize("name", list(CLOUDS))
def test_knn_and_order_are_exact(name, k):
    dev = cuda_or_skip()
    from paper_1603_04100_gb300 import api
    p = np.ascontiguousarray(CLOUDS[name]())
    pt = torch.from_numpy(p).to(dev)
    nbr, order = api.knn(pt, k, want_order=True)
    np.testing.assert_array_equal(nbr.cpu().numpy(), oracle.knn_brute(p, k))
    np.testing.assert_array_equal(order.cpu().numpy(), _order(p))
    # any cell size gives the same lists: thousands of candidates, or several rings
    e = float((p.max(0) - p.min(0)).max())
    for cell in (-3.0, -0.4, 0.6 * e):
        np.testing.assert_array_equal(api.knn(pt, k, cell_size=cell).cpu().numpy(), nbr.cpu().numpy())


@pytest.mark.parametrize("n", [3, 4, 33, 1025, 20000, 262147])
def test_row_order_at_tile_and_group_edges(n):
    dev = cuda_or_skip()
    from paper_1603_04100_gb300 import api
    p = I.random_sphere(n, 20 + n % 7)
    if n > 1000:
        p[500:900] = p[499]  # equal keys, ordered by index
    _, order = api.knn(torch.from_numpy(p).to(dev), 2, want_order=True)
    np.testing.assert_array_equal(order.cpu().numpy(), _order(p))
