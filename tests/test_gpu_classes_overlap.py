"""One step of a run with two size classes, of which one fills the device: the
other, a few larger cells, runs beside it (their cells are independent), with
the oracle's results."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from oracle import oracle as O
    from paper_2103_17238_gb300 import build as B
    from paper_2103_17238_gb300 import sdm

    B.build()
    O.build()
    torch.cuda.set_device(0)
    return O, sdm, torch


def _run(env, sizes):
    O, sdm, torch = env
    rng = np.random.default_rng(1)
    nc = len(sizes)
    cell = np.repeat(np.arange(nc, dtype=np.int32), sizes)
    n = len(cell)
    xi = rng.integers(1, 10**6, n).astype(np.int64)
    v = 4 / 3 * np.pi * np.exp(rng.uniform(np.log(3e-6), np.log(3e-4), n)) ** 3
    run = sdm.Run(sdm.make_config("geometric", dv=1e4, n_cells=nc, seed=1), n).set_attributes(xi, v, cell)
    return run, O.State(xi, v, cell, None, nc)


def _time(env, sizes):
    O, sdm, torch = env
    run, _ = _run(env, sizes)
    run.step(3)
    best = 1e9
    for _ in range(6):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        torch.cuda.synchronize()
        torch.cuda._sleep(3000000)
        a.record()
        for _ in range(40):
            run.step(1)
        b.record()
        torch.cuda.synchronize()
        best = min(best, a.elapsed_time(b) / 40)
    run.close()
    return best


@pytest.mark.parametrize("small,large", [([30] * 4096, [1000]), ([20] * 10000, [3000])])
def test_beside_each_other(env, small, large):
    O, sdm, torch = env
    run, st = _run(env, small + large)
    for k in (1, 1, 3):
        run.step(k)
    O.run(O.params("geometric", dv=1e4, seed=1), st, 0, 5)
    x, w = run.attributes()
    assert np.array_equal(x, st.xi) and np.array_equal(w, st.v)
    run.close()
    seen = []
    for _ in range(4):  # (new streams each time: which hardware queues they share is theirs to choose)
        seen.append((_time(env, small + large), _time(env, small), _time(env, large)))
        if seen[-1][0] < 0.9 * (seen[-1][1] + seen[-1][2]):  # one after the other: 0.99 and more
            return
    assert False, seen
