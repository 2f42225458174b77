"""Attributes given with the cells in no order: sorted on the device.

Within a cell super-droplets keep increasing id, so a run set from shuffled
input steps exactly as one set from the same super-droplets in (cell, id)
order.  Sizes lie at the edges of the sort's tiles (4096 keys) and of its
digits (one, two and three passes of 8 bits)."""
import numpy as np
import pytest

from paper_2103_17238_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n, n_cells", [(2, 2), (255, 3), (4095, 255), (4096, 256), (4097, 257), (50001, 65535),
                                        (70001, 70000)])
@pytest.mark.parametrize("on_device", [False, True])
def test_unsorted_cells(n, n_cells, on_device):
    torch = pytest.importorskip("torch")
    from paper_2103_17238_gb300 import sdm

    rng = np.random.default_rng(n)
    cell = rng.integers(-1, n_cells, n).astype(np.int32)
    cell[:2] = n_cells - 1, 0  # never in order
    xi, v = I.lognormal_sample(n, 1e3 * n, I.LOGNORMAL_RADIUS, I.LOGNORMAL_SIGMA)
    xi = xi + rng.integers(0, 1000, n)
    order = np.argsort(np.where(cell < 0, n_cells, cell), kind="stable")

    def final(xi, v, cell):
        if on_device:
            xi, v, cell = (torch.as_tensor(a, device="cuda") for a in (xi, v, cell))
        run = sdm.Run(sdm.make_config("golovin", dv=1e-6, n_cells=n_cells, seed=3), n)
        run.set_attributes(xi, v, cell)
        first = run.attributes()
        _, c = run.positions(want_z=False)
        run.step(3)
        out = run.attributes()
        run.close()
        return first, c, out

    (x0, v0), c, (x, w) = final(xi, v, cell)
    assert np.array_equal(x0, xi) and np.array_equal(v0, v) and np.array_equal(c, cell)
    _, _, (xs, ws) = final(xi[order], v[order], cell[order])
    assert np.array_equal(x[order], xs) and np.array_equal(w[order], ws)
    assert n < 300 or not np.array_equal(x, xi)  # pairs collided
