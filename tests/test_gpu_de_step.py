"""The on-chip DE step against the oracle where its branches change: unaligned and odd-sized
populations, penalties of either sign, n_min, more counts than shared memory holds (the general
step), the largest population it takes, and odd populations in the batched level solve."""
import numpy as np
import pytest

import oracle
from gpu_helpers import gpu_dataset

pytestmark = pytest.mark.gpu


def _data(seed, n, F, K):
    rng = np.random.Generator(np.random.PCG64(88_000 + seed))
    X = (np.floor(rng.random((n, F)) * 400) / 400).astype(np.float32)
    return X, rng.integers(0, K, n).astype(np.uint8)


@pytest.mark.parametrize("P,depth,K,alpha,n_min,dither,off", [
    (4, 1, 2, 0.0, 1, False, 0), (5, 2, 3, 0.0, 1, True, 1), (101, 3, 5, 0.0, 40, False, 3),
    (256, 3, 2, 1.5, 1, True, 2), (33, 4, 7, -0.75, 25, False, 1), (128, 5, 4, 0.25, 1, False, 0),
    (64, 6, 3, 0.0, 3, True, 1), (200, 5, 60, 0.0, 1, False, 0)])
def test_step_bit_exact(P, depth, K, alpha, n_min, dither, off):
    import torch
    from paper_2311_06952_gb300 import deoct
    n, F, G = 700, 9, 5
    X, y = _data(P, n, F, K)
    ranks, nu = oracle.encode(X)
    ref = oracle.de_run(ranks, nu, y, K, depth=depth, P=P, G=G, alpha=alpha, n_min=n_min, seed=9, dither=dither)
    ctx = deoct.Context(0)
    ds = gpu_dataset(ctx, X, y, K, 2)
    m = 2 * ((1 << depth) - 1)
    buf = torch.empty(P * m + off, dtype=torch.float32, device="cuda")
    pop = buf[off:].view(P, m)
    prm = deoct.make_params(depth, P, G, alpha=alpha, n_min=n_min, seed=9,
                            flags=deoct.DEOCT_DITHER_M if dither else 0)
    _, _, f = deoct.deoct_fit_subtree(ctx, ds, prm, pop_out=pop)
    np.testing.assert_array_equal(pop.cpu().numpy().view(np.uint32), ref["pop"].view(np.uint32))
    assert f == ref["fit"][ref["best"]]
    ctx.close()


@pytest.mark.parametrize("P,K", [(37, 3), (101, 2)])
def test_odd_population_in_level_solves(P, K):
    from paper_2311_06952_gb300 import deoct
    n, F = 2500, 5
    X, y = _data(P + 7, n, F, K)
    ranks, nu = oracle.encode(X)
    ref = oracle.mh(ranks, nu, y, K, depth=4, horizon=2, P=P, G=6, seed=3)
    ctx = deoct.Context(0)
    ds = gpu_dataset(ctx, X, y, K, 2)
    out = deoct.deoct_fit_moving_horizon(
        ctx, ds, deoct.make_params(4, P, 6, seed=3, horizon=2, flags=deoct.DEOCT_BATCHED))
    np.testing.assert_array_equal(out["a"], ref["a"])
    np.testing.assert_array_equal(out["theta"], ref["theta"])
    np.testing.assert_array_equal(out["leaf_class"], ref["leaf_class"])
    ctx.close()


@pytest.mark.parametrize("G", [1, 2, 3, 7, 8, 9, 16, 19])
@pytest.mark.parametrize("P,depth", [(64, 2), (300, 4), (12, 3)])
def test_generation_graphs(G, P, depth):
    """Generation counts around the captured graphs' eight, on every step and evaluator kernel."""
    import torch
    from paper_2311_06952_gb300 import deoct
    n, F, K = 1500, 6, 3
    X, y = _data(G + P, n, F, K)
    ranks, nu = oracle.encode(X)
    ref = oracle.de_run(ranks, nu, y, K, depth=depth, P=P, G=G, seed=4)
    ctx = deoct.Context(0)
    ds = gpu_dataset(ctx, X, y, K, 2)
    pop = torch.empty((P, 2 * ((1 << depth) - 1)), dtype=torch.float32, device="cuda")
    for _ in range(2):
        _, _, f = deoct.deoct_fit_subtree(ctx, ds, deoct.make_params(depth, P, G, seed=4), pop_out=pop)
        np.testing.assert_array_equal(pop.cpu().numpy().view(np.uint32), ref["pop"].view(np.uint32))
        assert f == ref["fit"][ref["best"]]
    ctx.close()
