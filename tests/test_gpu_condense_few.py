"""Condensation of few cells of several hundred super-droplets: a block per cell
(up to 1216 cells of 257 to 1024 slots) gives the oracle's volumes bit for bit
and its water within the summation bound, and costs no more rounds one after
the other than cells of 256 do."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

U = 2.0**-53


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


@pytest.mark.parametrize("sizes", [[257], [1024], [0, 1, 258, 511, 512, 513, 767, 768, 769, 1023, 1024], [300] * 1216,
                                   [300] * 1217, [5] * 1215 + [1000], [256] * 40])
def test_parity(env, sizes):
    O, sdm, torch = env
    rng = np.random.default_rng(len(sizes))
    nc = len(sizes)
    cell = np.repeat(np.arange(nc, dtype=np.int32), sizes)
    n = len(cell)
    xi = rng.integers(1, 10**9, n).astype(np.int64)
    xi[rng.random(n) < 0.05] = 0
    v = 4 / 3 * np.pi * np.exp(rng.uniform(np.log(5e-7), np.log(2e-3), n)) ** 3
    G, s = np.full(nc, 1e-10), rng.uniform(-0.05, 0.05, nc)
    run = sdm.Run(sdm.make_config("geometric", dv=1.0, n_cells=nc, seed=1), n).set_attributes(xi, v, cell)
    st = O.State(xi.copy(), v.copy(), cell.copy(), None, nc)
    P = O.params("geometric", dv=1.0, seed=1)
    for f in (s, s, -s):  # a new field, a repeated one, another
        before = st.v.copy()
        got, want = run.condense(G, f, 1e-6), O.condense(P, st, G, f, 1e-6)
        assert np.array_equal(run.attributes()[1], st.v)
        bound = 2 * max(sizes) * U * np.bincount(cell, weights=xi * np.abs(st.v - before) * (1 + 1e-6), minlength=nc)
        assert np.all(np.abs(got - want) <= bound + 1e-300)
        run.condense(G, f, 1e-6, want_condensed=False)
        O.condense(P, st, G, f, 1e-6)
        assert np.array_equal(run.attributes()[1], st.v)
    run.close()


def test_time(env):
    seen = []
    for _ in range(4):
        seen.append(_times(env))
        if seen[-1][1000] < 1.4 * seen[-1][250]:  # a warp per cell: 2.0
            return
    assert False, seen


def _times(env):
    O, sdm, torch = env
    times = {}
    for per in (250, 1000):
        nc = 300
        n = nc * per
        run = sdm.Run(sdm.make_config("geometric", dv=1.0, n_cells=nc, seed=1), n)
        run.set_attributes(torch.full((n,), 1000, dtype=torch.int64, device="cuda"),
                           torch.full((n,), 1e-14, dtype=torch.float64, device="cuda"),
                           torch.arange(nc, dtype=torch.int32, device="cuda").repeat_interleave(per))
        G, s = np.full(nc, 1e-10), np.full(nc, 0.001)

        def calls(k):
            for _ in range(k):
                sdm.sdm_condensation_step(run.h, G, s, 1e-6, want_condensed=False, n_cells=nc)

        calls(10)
        best = 1e9
        for _ in range(5):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            torch.cuda.synchronize()
            torch.cuda._sleep(2000000)
            a.record()
            calls(40)
            b.record()
            torch.cuda.synchronize()
            best = min(best, a.elapsed_time(b))
        times[per] = best / 40
        run.close()
    return times
