"""The autotuner of the batched level solve where it still runs: sets too wide for the
bit-sliced evaluator, with levels long enough to pay for timing the candidate shapes."""
import numpy as np
import pytest

from gpu_helpers import gpu_dataset

pytestmark = pytest.mark.gpu


def test_autotuned_wide_level_solve_equals_plain():
    """48 features of 6e5 distinct values (20 bits), 128 trees, 270 generations: above the 2e10
    tree-sample evaluations a level from which shapes are timed.  The batched fit gives the plain
    per-node fit's tree, with evaluator launches beyond the generations' own."""
    from paper_2311_06952_gb300 import deoct
    n, F, K, P, G = 600_000, 48, 3, 128, 270
    assert n * P * (G + 1) >= 2e10
    rng = np.random.Generator(np.random.PCG64(31))
    X = rng.random((n, F)).astype(np.float32)
    y = ((X[:, 3] > 0.4).astype(int) + (X[:, 7] * X[:, 3] > 0.3) * (rng.random(n) < 0.9)).astype(np.uint8)
    outs, evals, sliced = [], [], []
    for flags in (0, deoct.DEOCT_BATCHED):
        ctx = deoct.Context(0)
        ds = gpu_dataset(ctx, X, y, K, 4)
        ctx.reset_stats()
        outs.append(deoct.deoct_fit_moving_horizon(ctx, ds, deoct.make_params(3, P, G, seed=5, horizon=2, flags=flags)))
        evals.append(ctx.stats()["eval_launches"])
        sliced.append(ctx.slice_stats()[0])
        ctx.close()
    for k in ("a", "theta", "kind", "node_fit", "leaf_class"):
        np.testing.assert_array_equal(outs[0][k], outs[1][k], err_msg=k)
    assert sliced == [0, 0]
    levels = 2  # roots of horizon 2; the last level is the exhaustive search
    assert evals[1] >= levels * (G + 1) + 3 * 4  # four candidates or more, three timings each
