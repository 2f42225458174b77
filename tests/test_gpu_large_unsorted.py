"""Cells in no order about 2^21 super-droplets, where the device sort goes from
tiles of 1024 to tiles of 4096 keys (with a part-filled last one)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2103_17238_gb300 import build as B
    from paper_2103_17238_gb300 import sdm

    B.build()
    torch.cuda.set_device(0)
    return sdm, torch


@pytest.mark.parametrize("n", [(1 << 21) - 1, 1 << 21, (1 << 21) + 4097])
@pytest.mark.parametrize("n_cells", [200, 70001])
def test_layout(env, n, n_cells):
    """The state comes back by id, the cells too, and a step equals that of the
    same super-droplets given in cell order."""
    sdm, torch = env
    rng = np.random.default_rng(n_cells + n)
    cell = rng.integers(-1, n_cells, n).astype(np.int32)
    xi = rng.integers(0, 10**6, n).astype(np.int64)
    v = 4 / 3 * np.pi * np.exp(rng.uniform(np.log(2e-6), np.log(2e-4), n)) ** 3
    order = np.argsort(np.where(cell < 0, n_cells, cell), kind="stable")
    runs = []
    for p in (np.arange(n), order):
        r = sdm.Run(sdm.make_config("golovin", dv=1e2, n_cells=n_cells, seed=3), n)
        r.set_attributes(*(torch.as_tensor(a[p], device="cuda") for a in (xi, v, cell)))
        x, w = r.attributes()
        assert np.array_equal(x, xi[p]) and np.array_equal(w, v[p])
        assert np.array_equal(r.positions(want_z=False)[1], cell[p])
        r.step(1)
        runs.append(r.attributes())
        r.close()
    assert np.array_equal(runs[0][0][order], runs[1][0]) and np.array_equal(runs[0][1][order], runs[1][1])
    assert int((runs[0][0] != xi).sum()) > 0
