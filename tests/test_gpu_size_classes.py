"""Cells about the size classes' edges against the oracle, bit for bit, in the numbers that
choose a kernel: few cells of 129 to 512 SDs (a block each), many (a warp each, the class of
320), and small cells that join the next class's launch; one step per call and fused."""
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
    return O, sdm


MIXES = {
    "few": [256, 257, 319, 320, 321, 511, 512],
    "edge of few": [320] * 304 + [512] * 3,
    "many of 320": [257, 318, 319, 320] * 100 + [321] * 2,
    "many of 512": [321, 512] * 310,
    "folded": [2, 3, 63, 64, 65, 127, 128, 129, 255] * 40,
}


@pytest.mark.parametrize("mix", MIXES)
@pytest.mark.parametrize("kernel,dv", [("golovin", 1e0), ("geometric", 1e-3)])
def test_size_classes(env, mix, kernel, dv):
    O, sdm = env
    rng = np.random.default_rng(len(MIXES[mix]))
    sizes = MIXES[mix]
    cell = np.repeat(np.arange(len(sizes), dtype=np.int32), sizes)
    n = len(cell)
    xi = np.where(rng.random(n) < 0.3, 1000, rng.integers(1, 10**9, n)).astype(np.int64)
    xi[rng.random(n) < 0.05] = 0
    v = 4 / 3 * np.pi * np.exp(rng.uniform(np.log(2e-6), np.log(2e-3), n)) ** 3
    run = sdm.Run(sdm.make_config(kernel, dv=dv, n_cells=len(sizes), seed=7), n)
    run.set_attributes(xi, v, cell)
    for k in (1, 4, 1):
        run.step(k)
    gx, gv = run.attributes()
    run.close()
    st = O.State(xi.copy(), v.copy(), cell.copy(), None, len(sizes))
    O.run(O.params(kernel, dv=dv, seed=7), st, 0, 6)
    assert np.array_equal(gx, st.xi) and np.array_equal(gv, st.v)
    assert int((gx != xi).sum()) > 0
