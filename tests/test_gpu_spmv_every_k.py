"""The product at every K the operator can have: groups of four slots fixed at compile
time with 0 to 3 left over, 1 .. 8 right-hand sides, all three forms, ragged row counts,
against a float64 sum of the same stored weights.  Bounds: the terms' rounding, (K + 6)
units of the sum of magnitudes."""
from __future__ import annotations

import numpy as np
import pytest

from tests.gpu_util import cuda_or_skip, operator_from_rows

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k", range(1, 32))
@pytest.mark.parametrize("mode", ["f64", "f32", "hilo"])
def test_every_k_equals_the_sum(k, mode):
    dev = cuda_or_skip()
    from paper_1603_04100_gb300 import api
    n = 419
    rng = np.random.default_rng(100 + k)
    nbr = rng.integers(0, n, (n, k)).astype(np.int32)
    op = operator_from_rows(nbr, rng.standard_normal((n, k + 1)), api.FP64 if mode == "f64" else api.FP32_REFINE, dev)
    w = op.rows("val").astype(np.float64)
    if mode == "hilo":
        w = w + op.rows("val_lo").astype(np.float64)
    unit = 2.0 ** -24 if mode == "f32" else 2.0 ** -53
    const = {"f64": api.SPMV_F64, "f32": api.SPMV_F32, "hilo": api.SPMV_F64_HILO}[mode]
    dt = np.float32 if mode == "f32" else np.float64
    for q in range(1, 9):
        x = rng.standard_normal((n, q)).astype(dt)
        y = api.spmv(op, torch.from_numpy(x).to(dev), mode=const, sigma=0.75, alpha=-1.5)
        x64 = x.astype(np.float64)
        xj = x64[nbr]
        if mode == "f32":
            lx = (w[:, 1:, None] * (xj - x64[:, None, :])).sum(1)
            size = (np.abs(w[:, 1:, None]) * (np.abs(xj) + np.abs(x64[:, None, :]))).sum(1)
        else:
            lx = w[:, :1] * x64 + (w[:, 1:, None] * xj).sum(1)
            size = np.abs(w[:, :1]) * np.abs(x64) + (np.abs(w[:, 1:, None]) * np.abs(xj)).sum(1)
        want = -1.5 * (0.75 * x64 - lx)
        bound = 2 * (k + 6) * unit * 1.5 * (0.75 * np.abs(x64) + size)
        got = y.cpu().numpy().astype(np.float64)
        assert np.all(np.abs(got - want) <= bound), (q, float(np.max(np.abs(got - want) / bound)))
