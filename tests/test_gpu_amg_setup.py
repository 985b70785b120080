"""The multigrid set-up at the edges of its kernels: coarsest levels around the
panel (32) and block (64) widths of the blocked inversion up to its largest size,
and coarsening at every width of the per-lane entry lists, against the oracle's
hierarchy (oracle/amg.py) and numpy's inverse.  Bounds: those of a Gauss-Jordan
inverse in FP32 and of one refined in FP64, 4 n u cond(A), and FP64 sums in another
order, 64 ulps of the row."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
from oracle import amg as OA
from paper_1603_04100_gb300 import inputs as I
from tests.gpu_util import cuda_or_skip, operator_from_rows

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _operator(n, k, seed):
    pts = I.morton_sorted(I.random_sphere(n, seed))
    nbr = oracle.knn_grid(pts, k)
    val, st, _, _ = oracle.assemble(pts, nbr)
    assert int(st.max()) == 0
    return nbr, val


@pytest.mark.parametrize("n,k", [(13, 8), (31, 12), (32, 12), (33, 12), (64, 16), (65, 16), (97, 16), (129, 20),
                                 (257, 20), (448, 24), (511, 20), (512, 20), (513, 20), (4096, 20)])
def test_coarsest_inverse_at_every_panel_and_block_edge(n, k):
    dev = cuda_or_skip()
    from paper_1603_04100_gb300 import api
    nbr, val = _operator(n, k, 70)
    H = api.amg_setup(operator_from_rows(nbr, val, api.FP64, dev), 1.0)
    assert H.info(0).status == 0
    Ac = OA.hierarchy(val, nbr, 1.0)[-1].dense()
    nc = Ac.shape[0]
    want, cond = np.linalg.inv(Ac), np.linalg.cond(Ac)
    for fp64, u in ((False, 2.0 ** -24), (True, 2.0 ** -53)):
        X = H.coarsest_inverse(fp64=fp64).astype(np.float64)
        assert np.abs(Ac @ X - np.eye(nc)).max() <= 4 * nc * u * cond
        assert np.linalg.norm(X - want) / np.linalg.norm(want) <= 4 * nc * u * cond


def test_singular_coarsest_level_is_reported():
    dev = cuda_or_skip()
    from paper_1603_04100_gb300 import _lib as LB
    from paper_1603_04100_gb300 import api
    nbr, val = _operator(200, 12, 71)
    H = api.amg_setup(operator_from_rows(nbr, np.zeros_like(val), api.FP64, dev), 0.0)  # the zero matrix
    assert H.info(0).status == LB.EDEGENERATE


@pytest.mark.parametrize("prec_name", ["FP64", "FP32_REFINE"])
@pytest.mark.parametrize("n,k", [(515, 15), (1001, 12), (2001, 23), (4097, 31), (33000, 16)])
def test_coarsening_at_every_list_width(n, k, prec_name):
    dev = cuda_or_skip()
    from paper_1603_04100_gb300 import api
    nbr, val = _operator(n, k, 72)
    H = api.amg_setup(operator_from_rows(nbr, val, getattr(api, prec_name), dev), 1.0)
    levels = OA.hierarchy(val, nbr, 1.0)
    assert H.levels == len(levels)
    width = 0
    for lv in range(1, len(levels)):
        ref = levels[lv]
        cnt, col, v64, v32, dinv = H.level_rows(lv)
        want_cnt = np.bincount(ref.rows, minlength=ref.n)
        width = max(width, int(want_cnt.max()))
        assert np.array_equal(cnt, want_cnt)
        got_cols = np.concatenate([col[r, :cnt[r]] for r in range(ref.n)])
        got = np.concatenate([v64[r, :cnt[r]] for r in range(ref.n)])
        assert np.array_equal(got_cols, ref.cols)
        scale = np.zeros(ref.n)
        np.add.at(scale, ref.rows, np.abs(ref.vals))
        assert np.all(np.abs(got - ref.vals) <= 64 * np.finfo(np.float64).eps * scale[ref.rows])
        np.testing.assert_allclose(dinv, ref.d, rtol=2 ** -22, atol=0)
        pad = np.arange(col.shape[1])[None, :] >= cnt[:, None]
        assert np.all(v64[pad] == 0.0) and np.all(v32[pad] == 0.0)
        assert np.array_equal(col[pad], np.broadcast_to(np.arange(ref.n)[:, None], col.shape)[pad])
    assert H.info(0).width_max == width
