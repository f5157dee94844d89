"""The depth-1 search's integer ordering of candidates against the oracle: penalties from none
to past the integers' resolution in doubles, n_min, ties, many classes."""
import numpy as np
import pytest

import oracle
from gpu_helpers import gpu_dataset, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("alpha", [0.0, 0.25, float(2**49), float(2**51), 1e300])
@pytest.mark.parametrize("n,F,K,n_min", [(1, 2, 2, 1), (300, 4, 3, 1), (5000, 3, 2, 40), (2000, 6, 40, 7)])
def test_depth1(alpha, n, F, K, n_min):
    from paper_2311_06952_gb300 import deoct
    rng = np.random.Generator(np.random.PCG64(n + K))
    X = (np.floor(rng.random((n, F)) * 97) / 97).astype(np.float32)
    y = (rng.integers(0, K, n) * (X[:, 0] < 0.6)).astype(np.uint8)
    ranks, nu = oracle.encode(X)
    ctx = deoct.Context(0)
    ds = gpu_dataset(ctx, X, y, K, 2)
    for idx in (None, np.sort(rng.choice(n, max(1, n // 3), replace=False)).astype(np.int32)):
        ref = oracle.depth1(ranks, nu, y, K, n_min=n_min, alpha=alpha, idx=idx)
        got = deoct.deoct_depth1_search(ctx, ds, n_min=n_min, alpha=alpha, sample_idx=None if idx is None else to_dev(idx))
        assert tuple(got) == tuple(ref)
    ctx.close()
