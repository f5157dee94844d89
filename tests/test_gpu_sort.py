"""The encoder's segmented sort where it can go wrong: sizes around a sort tile (4096 keys), a
transpose block and a rank tile, one to many features, one distinct value, every value
distinct, runs of ties over tile borders, negative values, both zeros, infinities."""
import numpy as np
import pytest

import oracle
from gpu_helpers import to_dev, u16, u32

pytestmark = pytest.mark.gpu


def _values(kind, n, F, rng):
    if kind == "ties":
        return (np.floor(rng.random((n, F)) * 7) - 3).astype(np.float32)
    if kind == "one":
        return np.full((n, F), -2.5, np.float32)
    X = rng.normal(0, 1e3, (n, F)).astype(np.float32)
    if kind == "special":
        pick = rng.integers(0, 8, (n, F))
        for v, x in enumerate((np.inf, -np.inf, 0.0, -0.0, 1e-42)):
            X[pick == v] = x
    return X


@pytest.mark.parametrize("n", [1, 2, 31, 4095, 4096, 4097, 8193, 50_001])
@pytest.mark.parametrize("F,kind", [(1, "ties"), (3, "distinct"), (41, "special"), (161, "ties"), (256, "distinct"), (2, "one")])
def test_ranks(n, F, kind):
    import torch
    from paper_2311_06952_gb300 import deoct
    rng = np.random.Generator(np.random.PCG64(n * 7 + F))
    if n * F > 4_000_000:
        n = 4_000_000 // F
    X = _values(kind, n, F, rng)
    ranks, nu = oracle.encode(X)
    ctx = deoct.Context(0)
    for W in (2, 4, 0):
        if W == 2 and nu.max() > 65_536:
            continue
        if W:
            got, gnu = deoct.deoct_encode(ctx, to_dev(X), W)
        else:
            got, gnu, uniq, w = deoct.deoct_encode_auto(ctx, to_dev(X))
            assert w == (2 if nu.max() <= 65_536 else 4)
            for f in range(0, F, 50):
                np.testing.assert_array_equal(uniq[f, : nu[f]].cpu().numpy(), np.unique(X[:, f] + 0.0))
        r = u16(got) if got.dtype == torch.int16 else u32(got)
        np.testing.assert_array_equal(r[:, :n].astype(np.uint32), ranks)
        np.testing.assert_array_equal(u32(gnu), nu)
    ctx.close()
