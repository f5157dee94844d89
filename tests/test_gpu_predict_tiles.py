"""Prediction over row tiles and row by row against the oracle: row counts around a tile and a
16-byte piece, features on both sides of the rule between the two kernels, rows that start off
16 bytes, infinities and NaN, thresholds between, at and past float values."""
import numpy as np
import pytest

import oracle
from gpu_helpers import to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,F,depth,off", [
    (65_536, 28, 8, 0), (65_537, 28, 4, 0), (66_047, 7, 5, 0), (66_049, 3, 6, 0), (70_001, 5, 4, 1), (65_535, 28, 8, 0),
    (65_601, 64, 8, 0), (65_600, 65, 8, 0), (100_003, 1, 10, 0), (131_073, 80, 10, 0), (65_536, 28, 3, 0)])
def test_tiles(m, F, depth, off):
    import torch
    from paper_2311_06952_gb300 import deoct
    rng = np.random.Generator(np.random.PCG64(m + F + depth))
    B, K = (1 << depth) - 1, 5
    X = rng.normal(0, 2, (m, F)).astype(np.float32)
    X[rng.integers(0, m, 50), rng.integers(0, F, 50)] = np.inf
    X[rng.integers(0, m, 50), rng.integers(0, F, 50)] = -np.inf
    X[rng.integers(0, m, 50), rng.integers(0, F, 50)] = np.nan
    a = rng.integers(0, F + 1, B).astype(np.uint16)
    b = rng.normal(0, 1.5, B)
    b[::3] = X[rng.integers(0, m, len(b[::3])), 0].astype(np.float64)  # at data values
    b[1::7] += 1e-12                                                    # between neighbouring floats
    b[rng.integers(0, B, 2)] = (1e300, -1e300)
    b = np.where(np.isnan(b), 0.25, b)
    leaf = rng.integers(0, K, B + 1).astype(np.uint8)
    y = rng.integers(0, K, m).astype(np.uint8)
    buf = torch.empty(m * F + off, dtype=torch.float32, device="cuda")
    Xd = buf[off:].view(m, F)
    Xd.copy_(torch.from_numpy(X))
    ctx = deoct.Context(0)
    pred, ok = deoct.deoct_predict(ctx, Xd, to_dev(a), to_dev(b), depth, to_dev(leaf), y=to_dev(y))
    ref = oracle.predict(X, a, b, depth, leaf)
    np.testing.assert_array_equal(pred.cpu().numpy(), ref)
    assert int(ok.item()) == int((ref == y).sum())
    ctx.close()
