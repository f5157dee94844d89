"""Which evaluator a fit takes by default -- where the bit-sliced one was measured to be the
slower one it is not taken -- and that the choice changes no result, over the forms a fit
accepts: both rank widths, subsets, unaligned rows, few and many samples, wide sets, a level
solve of small nodes."""
import numpy as np
import pytest

from gpu_helpers import to_dev

pytestmark = pytest.mark.gpu


def _ds(n, F, K, bits, W, off=0, seed=0):
    from paper_2311_06952_gb300 import deoct
    rng = np.random.Generator(np.random.PCG64(n * 7 + F + bits + seed))
    pad = np.zeros((F, deoct.padded_ld(n, W) + off), np.uint16 if W == 2 else np.uint32)
    pad[:, :n] = rng.integers(0, 1 << bits, (F, n))
    y = np.minimum(rng.integers(0, K, n), rng.integers(0, K, n)).astype(np.uint8)
    y[pad[0, :n] > (1 << bits) // 2] = 0
    return deoct.DeviceDataset(to_dev(pad), W, to_dev(np.full(F, 1 << bits, np.uint32)), to_dev(y), n, F, K)


def _fit(ds, prm, mode, idx=None):
    import torch
    from paper_2311_06952_gb300 import deoct
    ctx = deoct.Context(0)
    ctx.set_eval_slicing(mode)
    pop = torch.empty((prm.pop, 2 * ((1 << prm.depth) - 1)), dtype=torch.float32, device="cuda")
    _, _, f = deoct.deoct_fit_subtree(ctx, ds, prm, pop_out=pop, sample_idx=idx)
    n = ctx.slice_stats()[0]
    ctx.close()
    return pop.cpu().numpy().view(np.uint32), f, n


@pytest.mark.parametrize("n,F,K,bits,W,P,depth,sliced", [
    (300_000, 38, 3, 20, 4, 128, 5, False),  # rows leave room for four trees a CTA: 627 us against 94
    (200, 30, 4, 17, 4, 128, 3, False),      # no planes: 21 against 10.7
    (1000, 30, 4, 17, 4, 128, 3, False),     # 14.2 against 10.9
    (20_000, 38, 2, 20, 4, 16, 3, False),    # 12.3 against 9.0
    (100_000, 24, 4, 16, 2, 128, 3, True),   # 18.4 against 25.4
    (300_000, 10, 2, 12, 2, 512, 4, True),   # 64 against 181
    (50_000, 8, 4, 10, 2, 128, 3, True)])    # 12.0 against 18.2
def test_measured_shapes_take_the_faster_evaluator(n, F, K, bits, W, P, depth, sliced):
    from paper_2311_06952_gb300 import deoct
    _, _, launches = _fit(_ds(n, F, K, bits, W), deoct.make_params(depth, P, 2, seed=1), 0)
    assert (launches > 0) == sliced


@pytest.mark.parametrize("n,F,K,bits,W,P,depth,off,subset", [
    (150, 5, 2, 7, 2, 16, 2, 0, False), (1025, 12, 9, 10, 2, 33, 3, 0, True), (5000, 30, 3, 17, 4, 64, 4, 1, False),
    (40_003, 20, 5, 15, 2, 100, 5, 3, True), (70_001, 40, 2, 16, 2, 48, 1, 0, False), (3000, 50, 4, 20, 4, 40, 5, 0, False)])
def test_the_choice_changes_no_result(n, F, K, bits, W, P, depth, off, subset):
    from paper_2311_06952_gb300 import deoct
    ds = _ds(n, F, K, bits, W, off)
    idx = to_dev(np.sort(np.random.default_rng(n).choice(n, n // 2, replace=False)).astype(np.int32)) if subset else None
    prm = deoct.make_params(depth, P, 9, seed=3)
    never, auto, always = (_fit(ds, prm, m, idx) for m in (-1, 0, 1))
    assert never[2] == 0
    for other in (auto, always):
        np.testing.assert_array_equal(other[0], never[0])
        assert other[1] == never[1]


@pytest.mark.parametrize("n,F,K,bits,W", [(1500, 24, 5, 12, 2), (60_000, 10, 3, 13, 2), (9000, 33, 4, 18, 4)])
def test_the_choice_changes_no_tree(n, F, K, bits, W):
    from paper_2311_06952_gb300 import deoct
    ds = _ds(n, F, K, bits, W, seed=1)
    out = []
    for mode in (-1, 0, 1):
        for flags in (0, deoct.DEOCT_BATCHED):
            ctx = deoct.Context(0)
            ctx.set_eval_slicing(mode)
            out.append(deoct.deoct_fit_moving_horizon(ctx, ds, deoct.make_params(5, 32, 9, seed=2, horizon=3, flags=flags)))
            assert mode == 0 or (ctx.slice_stats()[0] > 0) == (mode > 0)
            ctx.close()
    for o in out[1:]:
        for k in ("a", "theta", "kind", "node_fit", "leaf_class"):
            np.testing.assert_array_equal(o[k], out[0][k], err_msg=k)


def test_slicing_mode_is_checked():
    from paper_2311_06952_gb300 import deoct
    ctx = deoct.Context(0)
    for bad in (-2, 2):
        with pytest.raises(deoct.DeoctError):
            ctx.set_eval_slicing(bad)
    ctx.close()


@pytest.mark.parametrize("n,F,K,bits,W,P,depth,sliced", [
    (150_000, 24, 9, 20, 4, 931, 5, False),  # 814 us without planes against 381
    (480_000, 50, 3, 10, 2, 346, 4, False),  # 470 against 270
    (1_000_000, 10, 2, 16, 2, 512, 4, True)])
def test_measured_single_evaluations_take_the_faster_evaluator(n, F, K, bits, W, P, depth, sliced):
    import torch
    from paper_2311_06952_gb300 import deoct
    ds = _ds(n, F, K, bits, W)
    g = torch.Generator(device="cuda").manual_seed(n)
    B = (1 << depth) - 1
    a = torch.randint(0, F + 1, (P, B), generator=g, device="cuda").to(torch.int16)
    th = torch.randint(0, 1 << bits, (P, B), generator=g, device="cuda", dtype=torch.int32)
    out = []
    for mode in (-1, 0, 1):
        ctx = deoct.Context(0)
        ctx.set_eval_slicing(mode)
        counts, errors = deoct.deoct_eval_population(ctx, ds, a, th, depth)
        out.append((counts, errors, ctx.slice_stats()[0]))
        ctx.close()
    assert [o[2] for o in out] == [0, int(sliced), 1]
    for o in out[1:]:
        assert torch.equal(o[0], out[0][0]) and torch.equal(o[1], out[0][1])
