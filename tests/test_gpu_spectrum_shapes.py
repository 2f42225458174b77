"""Per-cell spectra where one cell holds most of the super-droplets, or all of
them: the oracle's values within the rounding of one binary64 addition per SD,
into host and device buffers, about the size where one cell goes from a block
to the whole device; and the time of a grid with one large cell."""
import numpy as np
import pytest

from paper_2103_17238_gb300 import inputs as I

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
    rng = np.random.default_rng(len(sizes) + sizes[-1])
    nc = len(sizes)
    cell = np.repeat(np.arange(nc, dtype=np.int32), sizes)
    n = len(cell)
    xi = rng.integers(1, 10**9, n).astype(np.int64)
    if n > 2:
        xi[rng.random(n) < 0.05] = 0
    v = 4 / 3 * np.pi * np.exp(rng.uniform(np.log(1e-6), np.log(3e-3), n)) ** 3
    run = sdm.Run(sdm.make_config("golovin", dv=1e6, n_cells=nc, seed=1), n).set_attributes(xi, v, cell)
    st = O.State(xi, v, cell, None, nc)
    return run, O.spectrum(O.params("golovin", dv=1e6, seed=1), st, I.R_EDGES, per_cell=True), n


@pytest.mark.parametrize("sizes", [[1], [2], [255], [256], [1024], [1025], [4095], [4096], [4097], [4098], [9001],
                                   [20] * 900 + [2048], [20] * 900 + [2049], [3] * 1536 + [2050], [3] * 1538 + [2050],
                                   [0, 1, 0, 30001], [7] * 3000 + [20000]])
def test_values(env, sizes):
    O, sdm, torch = env
    run, want, n = _run(env, sizes)
    out = torch.full((want.size,), np.nan, dtype=torch.float64, device="cuda")
    run.spectrum(I.R_EDGES, per_cell=True, out=out)
    host = run.spectrum(I.R_EDGES, per_cell=True)
    bound = 2 * (max(sizes) + 4) * 2.0**-53 * want
    assert np.all(np.abs(out.cpu().numpy().reshape(want.shape) - want) <= bound)
    assert np.all(np.abs(host - want) <= bound)
    assert want.max() > 0
    run.close()


def test_time_with_one_large_cell(env):
    O, sdm, torch = env
    run, want, n = _run(env, [20] * 10000 + [200000])
    out = torch.empty(want.size, dtype=torch.float64, device="cuda")
    times = []
    for _ in range(6):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        torch.cuda.synchronize()
        a.record()
        run.spectrum(I.R_EDGES, per_cell=True, out=out)
        b.record()
        torch.cuda.synchronize()
        times.append(a.elapsed_time(b))
    run.close()
    assert min(times) < 1.0, times  # ms: 2.0 with a warp per cell
