"""The bit-sliced evaluator through fits that are told to take it wherever it can run, and through
single evaluations large enough for it; every test asserts that it ran, and with how many digits a
threshold.  Ranks are drawn as such, with their n_p, so that small sets reach every digit
count, with planes in memory and without ("raw": the context's scratch is capped at what the
same fit holds on the other kernels, which leaves the planes no room)."""
import threading

import numpy as np
import pytest

import oracle
from gpu_helpers import gpu_dataset, to_dev, u32
from paper_2311_06952_gb300 import datagen

pytestmark = pytest.mark.gpu


def _rng(seed):
    return np.random.Generator(np.random.PCG64(91_000 + seed))


def _set(rng, n, F, K, bits, W):
    """Ranks of F features on n samples below n_p = 2^bits (the first feature) or a little less,
    with the least and the largest rank among them; labels of K classes."""
    from paper_2311_06952_gb300 import deoct
    nu = np.array([(1 << bits) - (f % 3 if bits > 2 else 0) for f in range(F)], np.uint32)
    ranks = np.stack([rng.integers(0, int(m), n) for m in nu]).astype(np.uint32)
    ranks[:, 0] = nu - 1
    ranks[:, n // 2] = 0
    y = rng.integers(0, K, n).astype(np.uint8)
    pad = np.zeros((F, deoct.padded_ld(n, W)), np.uint16 if W == 2 else np.uint32)
    pad[:, :n] = ranks
    ds = deoct.DeviceDataset(to_dev(pad), W, to_dev(nu), to_dev(y), n, F, K)
    return ranks, nu, y, ds


def _fit(ds, prm, raw):
    """One fit in a context of its own: (population, fitness, bit-sliced launches, digits)."""
    import torch
    from paper_2311_06952_gb300 import deoct
    ctx = deoct.Context(0)
    try:
        if raw:
            ctx.set_eval_config(S=512, TG=16)
            deoct.deoct_fit_subtree(ctx, ds, prm)
            ctx.set_eval_config()
            ctx.set_scratch_limit(ctx.memory()[0])
        else:  # as in a context that encoded the set: the planes' memory is there
            big = gpu_dataset(ctx, np.random.default_rng(0).random((20_000, 16)), np.zeros(20_000), 2, 2)
            del big
        ctx.set_eval_slicing(1)
        ctx.reset_stats()
        pop = torch.empty((prm.pop, 2 * ((1 << prm.depth) - 1)), dtype=torch.float32, device="cuda")
        _, _, f = deoct.deoct_fit_subtree(ctx, ds, prm, pop_out=pop)
        return (pop.cpu().numpy(), f) + ctx.slice_stats()
    finally:
        ctx.close()


def _check_fit(ranks, nu, y, K, ds, depth, P, G, raw, digits=None):
    from paper_2311_06952_gb300 import deoct
    ref = oracle.de_run(ranks, nu, y, K, depth=depth, P=P, G=G, seed=11)
    pop, f, launches, nd = _fit(ds, deoct.make_params(depth, P, G, seed=11), raw)
    np.testing.assert_array_equal(pop.view(np.uint32), ref["pop"].view(np.uint32))
    assert f == ref["fit"][ref["best"]]
    if digits == 0:
        assert launches == 0
    else:
        assert launches == G + 1 and (digits is None or nd == digits), (launches, nd)


@pytest.mark.parametrize("raw", [False, True])
@pytest.mark.parametrize("n", [1, 31, 33, 63, 64, 65, 1023, 1024, 1025, 2047, 3000])
@pytest.mark.parametrize("depth,K,P", [(1, 2, 17), (2, 3, 18), (3, 9, 16), (4, 2, 19), (5, 5, 21)])
def test_tile_edges(n, depth, K, P, raw):
    """Sample counts around a word, a word pair and a tile; tree counts off the multiples of four."""
    ranks, nu, y, ds = _set(_rng(n * 31 + depth), n, 5, K, 9, 2 if depth % 2 else 4)
    _check_fit(ranks, nu, y, K, ds, depth, P, 1, raw)


@pytest.mark.parametrize("raw", [False, True])
@pytest.mark.parametrize("depth,K", [(1, 2), (2, 9), (3, 2), (4, 9), (5, 2)])
@pytest.mark.parametrize("bits,F,W,digits", [(4, 20, 2, 1), (8, 20, 2, 2), (13, 20, 2, 3), (16, 20, 2, 4), (16, 30, 2, 5),
                                             (20, 23, 4, 6), (20, 28, 4, 7), (20, 33, 4, 8), (20, 36, 4, 10),
                                             (24, 30, 4, 12), (20, 45, 4, 0)])
def test_digit_counts(bits, F, W, digits, depth, K, raw):
    """Every digit count the kernel is built for, and sets too wide for it."""
    ranks, nu, y, ds = _set(_rng(bits * 64 + F), 1700, F, K, bits, W)
    _check_fit(ranks, nu, y, K, ds, depth, 16, 2, raw, digits)


@pytest.mark.parametrize("F,digits,past", [(12, 4, False), (28, 6, False), (40, 8, False), (28, 6, True)])
def test_single_evaluation_of_wide_ranks(F, digits, past):
    """2^27 tree-samples: the ranks are transposed in the launch, uint32, up to eight digits; with
    `past`, thresholds and ranks past the bound the launch is sized by (the general path)."""
    from paper_2311_06952_gb300 import deoct
    n, P, K, depth = 131_149, 1024, 3, 3
    rng = _rng(F + past)
    ranks, nu, y, ds = _set(rng, n, F, K, 24 if past else 17, 4)
    a, th = datagen.random_population(nu, P, depth, rng, allow_nosplit=True)
    th[0] = 0
    th[1] = np.where(a[1] > 0, nu[np.maximum(a[1].astype(int) - 1, 0)] - 1, 0)
    ctx = deoct.Context(0)
    ctx.set_eval_slicing(1)
    counts, errors = deoct.deoct_eval_population(ctx, ds, to_dev(a.astype(np.uint16)), to_dev(th.astype(np.uint32)), depth)
    got = ctx.slice_stats()
    ref = oracle.eval_counts_omp(ranks, y, K, a, th, depth)
    np.testing.assert_array_equal(u32(counts), ref)
    np.testing.assert_array_equal(u32(errors), oracle.fitness(ref, a, n)[1])
    assert got == (1, digits)
    ctx.close()


def test_contexts_fit_side_by_side():
    """Four threads, each with its own context and stream, encode and fit again and again: the
    same trees as alone, and all of them end."""
    import torch
    from paper_2311_06952_gb300 import deoct
    jobs = []
    for i, (n, F, K, depth) in enumerate([(3000, 6, 2, 4), (20_000, 9, 3, 3), (9000, 30, 5, 5), (70_000, 5, 2, 4)]):
        rng = _rng(500 + i)
        X = torch.from_numpy(rng.random((n, F)).astype(np.float32)).cuda()
        y = torch.from_numpy(rng.integers(0, K, n).astype(np.uint8)).cuda()
        jobs.append((X, y, K, deoct.make_params(depth, 32, 25, seed=i, horizon=3, flags=deoct.DEOCT_BATCHED)))

    def work(job, times, out):
        X, y, K, prm = job
        ctx = deoct.Context(0)
        ctx.set_eval_slicing(1)
        s = torch.cuda.Stream()
        with torch.cuda.stream(s):
            for _ in range(times):
                ds = deoct.encode_dataset(ctx, X, y, K, 0, stream=s)
                out.append(deoct.deoct_fit_moving_horizon(ctx, ds, prm, stream=s))
        out.append(ctx.slice_stats()[0])
        ctx.close()

    torch.cuda.synchronize()
    alone, together = [[] for _ in jobs], [[] for _ in jobs]
    for j, o in zip(jobs, alone):
        work(j, 1, o)
    threads = [threading.Thread(target=work, args=(j, 6, o), daemon=True) for j, o in zip(jobs, together)]
    for t in threads:
        t.start()
    for t in threads:
        t.join(timeout=120)
    assert not any(t.is_alive() for t in threads)
    for one, many in zip(alone, together):
        assert len(many) == 7 and many[-1] > 0
        for got in many[:-1]:
            for k in ("a", "theta", "kind", "node_fit", "leaf_class"):
                np.testing.assert_array_equal(got[k], one[0][k], err_msg=k)
