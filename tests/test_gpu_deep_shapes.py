"""Single evaluations in the shared-atomic mode (deep trees, many bins) against the oracle at
the launch shapes the chooser reaches: wide rows beside one CTA per SM, tiles of 128 samples,
fewer than 16 trees beside any tile, gathered and unaligned rows, populations off 16."""
import numpy as np
import pytest

import oracle
from gpu_helpers import to_dev, u32
from paper_2311_06952_gb300 import datagen

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,F,W,P,depth,K,subset,off", [
    (5000, 250, 4, 64, 6, 3, False, 0), (40_001, 250, 4, 17, 6, 3, False, 0), (6001, 200, 2, 150, 6, 2, True, 0),
    (9000, 12, 2, 40, 10, 5, False, 0), (30_000, 10, 2, 32, 8, 29, False, 0), (3000, 4, 4, 5, 10, 40, False, 0),
    (70_000, 30, 4, 7, 7, 2, True, 0), (33_333, 22, 4, 100, 6, 2, False, 1), (20_000, 7, 2, 33, 5, 90, True, 3),
    (100, 5, 2, 1, 6, 2, False, 0)])
def test_deep_evaluation(n, F, W, P, depth, K, subset, off):
    from paper_2311_06952_gb300 import deoct
    rng = np.random.Generator(np.random.PCG64(n + F + P))
    nu = np.full(F, 3000, np.uint32)
    ranks = rng.integers(0, 3000, (F, n)).astype(np.uint32)
    y = rng.integers(0, K, n).astype(np.uint8)
    a, th = datagen.random_population(nu, P, depth, rng, allow_nosplit=True)
    idx = np.sort(rng.choice(n, n // 2, replace=False)).astype(np.int32) if subset else None
    ld = deoct.padded_ld(n, W) + off  # off: rows that bulk copies cannot take
    pad = np.zeros((F, ld), np.uint16 if W == 2 else np.uint32)
    pad[:, :n] = ranks
    ds = deoct.DeviceDataset(to_dev(pad), W, to_dev(nu), to_dev(y), n, F, K)
    ctx = deoct.Context(0)
    counts, errors = deoct.deoct_eval_population(ctx, ds, to_dev(a.astype(np.uint16)), to_dev(th.astype(np.uint32)), depth,
                                                 sample_idx=None if idx is None else to_dev(idx))
    ref = oracle.eval_counts_omp(ranks, y, K, a, th, depth, idx=idx)
    np.testing.assert_array_equal(u32(counts), ref)
    np.testing.assert_array_equal(u32(errors), oracle.fitness(ref, a, n if idx is None else len(idx))[1])
    ctx.close()
