"""The product's paths: K fixed at compile time and at run time, wide and scalar loads of
1 .. 8 right-hand sides, all three forms, ragged row counts, against a float64 sum of the
same stored weights.  Bounds: the terms' rounding, (K + 6) units of the sum of magnitudes."""
from __future__ import annotations

import numpy as np
import pytest

from paper_1603_04100_gb300 import inputs as I
from tests.gpu_util import cuda_or_skip

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [33, 257, 4999])
@pytest.mark.parametrize("k", [12, 13, 16, 20, 24, 31])
@pytest.mark.parametrize("mode", ["f64", "f32", "hilo"])
def test_every_width_equals_the_sum(n, k, mode):
    dev = cuda_or_skip()
    from paper_1603_04100_gb300 import api
    p = torch.from_numpy(I.random_sphere(n, 5)).to(dev)
    op = api.assemble(p, api.knn(p, k), prec=api.FP64 if mode == "f64" else api.FP32_REFINE)
    col = op.rows("col").astype(np.int64)
    w = op.rows("val").astype(np.float64)
    if mode == "hilo":
        w = w + op.rows("val_lo").astype(np.float64)
    unit = 2.0 ** -24 if mode == "f32" else 2.0 ** -53
    sigma, alpha, beta = 0.75, -1.5, 0.5
    const = {"f64": api.SPMV_F64, "f32": api.SPMV_F32, "hilo": api.SPMV_F64_HILO}[mode]
    rng = np.random.default_rng(n + k)
    dt = np.float32 if mode == "f32" else np.float64
    for q in range(1, 9):
        x = rng.standard_normal((n, q)).astype(dt)
        y0 = rng.standard_normal((n, q)).astype(dt)
        y = torch.from_numpy(y0.copy()).to(dev)
        api.spmv(op, torch.from_numpy(x).to(dev), mode=const, sigma=sigma, alpha=alpha, beta=beta, y=y)
        x64, y64 = x.astype(np.float64), y0.astype(np.float64)
        xj = x64[col]                                            # [n][k][q]
        if mode == "f32":
            lx = (w[:, 1:, None] * (xj - x64[:, None, :])).sum(1)
            size = (np.abs(w[:, 1:, None]) * (np.abs(xj) + np.abs(x64[:, None, :]))).sum(1)
        else:
            lx = w[:, :1] * x64 + (w[:, 1:, None] * xj).sum(1)
            size = np.abs(w[:, :1]) * np.abs(x64) + (np.abs(w[:, 1:, None]) * np.abs(xj)).sum(1)
        want = alpha * (sigma * x64 - lx) + beta * y64
        bound = 2 * (k + 6) * unit * (abs(alpha) * (sigma * np.abs(x64) + size) + beta * np.abs(y64))
        got = y.cpu().numpy().astype(np.float64)
        assert np.all(np.abs(got - want) <= bound), (q, float(np.max(np.abs(got - want) / bound)))
