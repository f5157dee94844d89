"""Memory a fit can do without (the planes of the bit-sliced evaluator) under a context's
scratch cap: a fit that runs without it runs with it too, again in the same context, with the
same result and within the cap."""
import numpy as np
import pytest

from gpu_helpers import gpu_dataset

pytestmark = pytest.mark.gpu

N, F, K, LEVELS = 40_000, 8, 3, 5000
PLANES = (N + 1023) // 1024 * (F * 13 + K + 2) * 128  # of the whole set: 13 bits hold LEVELS ranks


@pytest.fixture(scope="module")
def data():
    from paper_2311_06952_gb300 import deoct
    rng = np.random.Generator(np.random.PCG64(4711))
    X = (np.floor(rng.random((N, F)) * LEVELS) / LEVELS).astype(np.float32)
    y = np.where(X[:, 0] + 0.4 * rng.random(N) < 0.6, 0, rng.integers(1, K, N)).astype(np.uint8)
    enc = deoct.Context(0)  # the fits' contexts hold nothing of the encoder's
    ds = gpu_dataset(enc, X, y, K, 2)
    yield ds
    enc.close()


def _subtree(ctx, ds):
    from paper_2311_06952_gb300 import deoct
    return deoct.deoct_fit_subtree(ctx, ds, deoct.make_params(3, 32, 4, seed=2))


def _horizon(flags):
    def fit(ctx, ds):
        from paper_2311_06952_gb300 import deoct
        prm = deoct.make_params(4, 32, 4, seed=2, horizon=2, flags=deoct.DEOCT_BATCHED if flags else 0)
        out = deoct.deoct_fit_moving_horizon(ctx, ds, prm)
        return out["a"], out["theta"], out["node_fit"]
    return fit


def _with(ds, fit, cap, forced, times=1):
    from paper_2311_06952_gb300 import deoct
    ctx = deoct.Context(0)
    try:
        if forced:  # a forced launch shape keeps the fit off the bit-sliced evaluator and its planes
            ctx.set_eval_config(S=512, TG=32)
        else:  # and this on it
            ctx.set_eval_slicing(1)
        ctx.set_scratch_limit(cap)
        for _ in range(times):
            out = fit(ctx, ds)
            assert cap == 0 or ctx.memory()[0] - 4 <= cap
        return out, ctx.memory()[0]
    finally:
        ctx.close()


def _same(got, want):
    for g, w in zip(got, want):
        np.testing.assert_array_equal(np.asarray(g), np.asarray(w))


@pytest.mark.parametrize("above", [16, 24, 48, 64, 200, 400])
def test_subtree_fit_with_a_cap_a_little_above_the_planes(data, above):
    want, held = _with(data, _subtree, 0, True)
    assert held < 16 * 1024  # what the fit needs without planes
    got, _ = _with(data, _subtree, PLANES + above * 1024, False, times=2)
    _same(got, want)


@pytest.mark.parametrize("batched", [False, True])
def test_horizon_fit_with_the_cap_that_suffices_without_planes(data, batched):
    want, held = _with(data, _horizon(batched), 0, True)
    _same(_with(data, _horizon(batched), held, True)[0], want)
    got, _ = _with(data, _horizon(batched), held, False, times=2)
    _same(got, want)


def test_engine_jobs_take_no_memory_for_planes(data):
    """A level solve whose generations run in a shared engine's launches, which read no planes,
    takes no memory for them (and so builds none)."""
    from paper_2311_06952_gb300 import deoct
    want, plain = _with(data, _horizon(True), 0, True)
    eng = deoct.Engine(0)
    ctx = deoct.Context(0)
    try:
        ctx.attach_engine(eng)
        got = _horizon(True)(ctx, data)
        held = ctx.memory()[0]
    finally:
        ctx.close()
        eng.close()
    _same(got, want)
    assert held < plain + PLANES // 2, (held, plain, PLANES)


@pytest.mark.parametrize("P,depth", [(8, 2), (16, 6)])
def test_a_fit_on_the_other_kernels_reads_back_only_its_result(P, depth):
    """Fewer than 16 trees and depth 6 keep a fit off the bit-sliced evaluator: it then has no
    use for n_p on the host (a wait for the stream), and holds no pinned memory for it."""
    from paper_2311_06952_gb300 import deoct
    from gpu_helpers import to_dev
    n, F = 500, 250
    rng = np.random.Generator(np.random.PCG64(P + depth))
    pad = np.zeros((F, deoct.padded_ld(n, 2)), np.uint16)
    pad[:, :n] = rng.integers(0, 50, (F, n))
    ds = deoct.DeviceDataset(to_dev(pad), 2, to_dev(np.full(F, 50, np.uint32)), to_dev(rng.integers(0, 2, n).astype(np.uint8)),
                             n, F, 2)
    ctx = deoct.Context(0)
    deoct.deoct_fit_subtree(ctx, ds, deoct.make_params(depth, P, 2, seed=1))
    assert ctx.memory()[1] < 4 * F
    ctx.close()
