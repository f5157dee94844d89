"""The bit-sliced evaluator (depth 1 to 5) against the oracle where it can go wrong: tile and
word edges, digit counts from one bit to the widest ranks, feature counts up to the most the
thermometer rows take and past it, classes that share tiles, thresholds past the rows' range
(the in-kernel general path), unaligned rows, subsets, and the planes of fits."""
import numpy as np
import pytest

import oracle
from gpu_helpers import gpu_dataset, to_dev, u32
from paper_2311_06952_gb300 import datagen

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def c():
    from paper_2311_06952_gb300 import deoct
    ctx = deoct.Context(0)
    yield ctx
    ctx.close()


def _rng(seed):
    return np.random.Generator(np.random.PCG64(77_000 + seed))


def _check(c, ds, ranks, y, K, a, th, depth, idx=None):
    from paper_2311_06952_gb300 import deoct
    ref = oracle.eval_counts(ranks, y, K, a, th, depth, idx=idx)
    counts, errors = deoct.deoct_eval_population(c, ds, to_dev(a.astype(np.uint16)), to_dev(th.astype(np.uint32)), depth,
                                                 sample_idx=None if idx is None else to_dev(idx))
    n = len(y) if idx is None else len(idx)
    np.testing.assert_array_equal(u32(counts), ref)
    _, ref_err, _, _ = oracle.fitness(ref, a, n)
    np.testing.assert_array_equal(u32(errors), ref_err)


@pytest.mark.parametrize("n", [1, 31, 33, 63, 64, 65, 1023, 1024, 1025, 2047, 3000])
@pytest.mark.parametrize("depth,K,P", [(1, 2, 193), (2, 3, 195), (3, 9, 200), (4, 2, 258), (5, 5, 192)])
def test_tile_edges(c, n, depth, K, P):
    """Sample counts around a word, a word pair and a tile; tree counts off the multiples of four."""
    rng = _rng(n * 31 + depth)
    X = (np.floor(rng.random((n, 5)) * 300) / 300).astype(np.float32)
    y = rng.integers(0, K, n).astype(np.uint8)
    ranks, nu = oracle.encode(X)
    a, th = datagen.random_population(nu, P, depth, rng, allow_nosplit=True)
    for W in (2, 4):
        _check(c, gpu_dataset(c, X, y, K, W), ranks, y, K, a, th, depth)


@pytest.mark.parametrize("F,levels,W", [(1, 2, 2), (3, 1, 4), (7, 60_000, 2), (30, 200_000, 4), (48, 50_000, 2), (60, 70_000, 4),
                                        (200, 30, 2)])
def test_digit_counts(c, F, levels, W):
    """Rank ranges and feature counts from one digit to the launches that fall to the other kernels."""
    rng = _rng(F)
    n, K, P, depth = 70_001, 4, 200, 3
    X = (np.floor(rng.random((n, F)) * levels) / levels).astype(np.float32)
    y = rng.integers(0, K, n).astype(np.uint8)
    ranks, nu = oracle.encode(X)
    a, th = datagen.random_population(nu, P, depth, rng, allow_nosplit=True)
    th[0] = 0
    th[1] = np.where(a[1] > 0, np.asarray(nu)[np.maximum(a[1] - 1, 0)] - 1, 0)
    _check(c, gpu_dataset(c, X, y, K, W), ranks, y, K, a, th, depth)


@pytest.mark.parametrize("W,top", [(2, 65_535), (2, (1 << 24) - 1), (4, (1 << 24) - 1)])
def test_thresholds_past_the_set(c, W, top):
    """A view of a larger encoded set (ranks past the view's size) and thresholds past n_p."""
    from paper_2311_06952_gb300 import deoct
    rng = _rng(W + top)
    n, F, K, P, depth, part = 30_000, 6, 3, 210, 4, 1500
    X = rng.random((n, F)).astype(np.float32)
    y = rng.integers(0, K, n).astype(np.uint8)
    ranks, nu = oracle.encode(X)
    a, th = datagen.random_population(nu, P, depth, rng, allow_nosplit=True)
    th[::7] = np.where(a[::7] > 0, top, 0)
    full = gpu_dataset(c, X, y, K, W)
    view = deoct.DeviceDataset(full.ranks, W, full.n_unique, full.labels, part, F, K)
    _check(c, view, ranks[:, :part], y[:part], K, a, th, depth)


@pytest.mark.parametrize("n,K,depth,subset", [(1500, 2, 2, False), (9000, 3, 3, True), (20_001, 10, 3, False),
                                              (33_000, 2, 4, True), (12_345, 29, 5, False)])
def test_fit_planes(c, n, K, depth, subset):
    """A fit's planes (ordered by class when there are enough tiles) give the oracle's trajectory,
    also where the context's scratch limit leaves them no memory."""
    import torch
    from paper_2311_06952_gb300 import deoct
    rng = _rng(n + K)
    F, P, G = 6, 48, 3
    X = (np.floor(rng.random((n, F)) * 5000) / 5000).astype(np.float32)
    y = np.minimum(rng.integers(0, K, n), rng.integers(0, K, n)).astype(np.uint8)
    ranks, nu = oracle.encode(X)
    idx = np.sort(rng.choice(n, n * 2 // 3, replace=False)).astype(np.int32) if subset else None
    ref = oracle.de_run(ranks, nu, y, K, depth=depth, P=P, G=G, seed=5, idx=idx)
    prm = deoct.make_params(depth, P, G, seed=5)
    ds = gpu_dataset(c, X, y, K, 2)
    for limited in (False, True):
        ctx = deoct.Context(0)
        if limited:
            ctx.set_scratch_limit(P * ((1 << depth) * (K + 5) * 4 + 2 * 2 * (1 << depth) * 4 + 64) + 65_536)
        pop = torch.empty((P, 2 * ((1 << depth) - 1)), dtype=torch.float32, device="cuda")
        _, _, f = deoct.deoct_fit_subtree(ctx, ds, prm, pop_out=pop, sample_idx=None if idx is None else to_dev(idx))
        np.testing.assert_array_equal(pop.cpu().numpy().view(np.uint32), ref["pop"].view(np.uint32))
        assert f == ref["fit"][ref["best"]]
        ctx.close()


@pytest.mark.parametrize("n,P,W,depth,K", [(32_768, 4096, 2, 3, 2), (32_769, 4099, 4, 2, 3), (33_791, 4096, 2, 4, 5),
                                           (700_001, 195, 4, 1, 4)])
def test_one_large_evaluation(c, n, P, W, depth, K):
    """Single evaluations large enough for the kernel to transpose the ranks itself."""
    rng = _rng(n)
    X = (np.floor(rng.random((n, 6)) * 9000) / 9000).astype(np.float32)
    y = rng.integers(0, K, n).astype(np.uint8)
    ranks, nu = oracle.encode(X)
    a, th = datagen.random_population(nu, P, depth, rng, allow_nosplit=True)
    _check(c, gpu_dataset(c, X, y, K, W), ranks, y, K, a, th, depth)


@pytest.mark.parametrize("W,top", [(2, 65_535), (2, (1 << 24) - 1), (4, (1 << 24) - 1)])
def test_large_evaluation_past_the_set(c, W, top):
    """The same on a view of a larger encoded set with thresholds past it: the general path."""
    from paper_2311_06952_gb300 import deoct
    rng = _rng(W + top + 1)
    n, F, K, P, depth, part = 30_000, 6, 3, 90_000, 2, 1501
    X = rng.random((n, F)).astype(np.float32)
    y = rng.integers(0, K, n).astype(np.uint8)
    ranks, nu = oracle.encode(X)
    a, th = datagen.random_population(nu, P, depth, rng, allow_nosplit=True)
    th[::7] = np.where(a[::7] > 0, top, 0)
    full = gpu_dataset(c, X, y, K, W)
    view = deoct.DeviceDataset(full.ranks, W, full.n_unique, full.labels, part, F, K)
    _check(c, view, ranks[:, :part], y[:part], K, a, th, depth)
