"""A fit runs its generations as CUDA graphs.  What other threads do meanwhile -- close contexts,
synchronise the device, free memory -- does not end it, and its result is the same."""
import threading

import numpy as np
import pytest

from gpu_helpers import to_dev

pytestmark = pytest.mark.gpu


def _ds(n, F, K):
    from paper_2311_06952_gb300 import deoct
    rng = np.random.Generator(np.random.PCG64(n))
    pad = np.zeros((F, deoct.padded_ld(n, 2)), np.uint16)
    pad[:, :n] = rng.integers(0, 500, (F, n))
    return deoct.DeviceDataset(to_dev(pad), 2, to_dev(np.full(F, 500, np.uint32)),
                               to_dev(rng.integers(0, K, n).astype(np.uint8)), n, F, K)


def _close_contexts():
    from paper_2311_06952_gb300 import deoct
    deoct.Context(0).close()


def _synchronise():
    import torch
    torch.cuda.synchronize()


def _scratch():
    from paper_2311_06952_gb300 import deoct
    ctx = deoct.Context(0)
    _fit(ctx, _fit.ds, 3)
    ctx.release_scratch()
    ctx.close()


def _fit(ctx, ds, G, horizon=False):
    import torch
    from paper_2311_06952_gb300 import deoct
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        if horizon:
            prm = deoct.make_params(4, 32, G, seed=3, horizon=2, flags=deoct.DEOCT_BATCHED)
            out = deoct.deoct_fit_moving_horizon(ctx, ds, prm, stream=s)
            return out["a"], out["theta"], out["node_fit"]
        return deoct.deoct_fit_subtree(ctx, ds, deoct.make_params(3, 32, G, seed=3), stream=s)


@pytest.mark.parametrize("horizon", [False, True])
@pytest.mark.parametrize("other", [_close_contexts, _synchronise, _scratch])
def test_fit_beside_another_thread(other, horizon):
    from paper_2311_06952_gb300 import deoct
    ds = _fit.ds = _ds(3000, 6, 3)
    ctx = deoct.Context(0)
    want = _fit(ctx, ds, 11, horizon)
    stop, failed = threading.Event(), []

    def disturb():
        try:
            while not stop.is_set():
                other()
        except BaseException as e:  # noqa: BLE001
            failed.append(e)

    threads = [threading.Thread(target=disturb, daemon=True) for _ in range(2)]
    for t in threads:
        t.start()
    try:
        for _ in range(150):
            for g, w in zip(_fit(ctx, ds, 11, horizon), want):
                np.testing.assert_array_equal(np.asarray(g), np.asarray(w))
    finally:
        stop.set()
        for t in threads:
            t.join(timeout=60)
    assert not failed and not any(t.is_alive() for t in threads)
    ctx.close()
