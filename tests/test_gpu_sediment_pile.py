"""Super-droplets that pile up in a few cells: a step that finds more arrivals
in one cell than a block merges is taken by the sort, from the same state, as
are the next sixteen; then the cells take them one by one again.  Cells,
heights and states are the oracle's throughout, bit for bit; and a pile of
64,000 costs what the sort costs, not what one block's merge of it would."""
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


def _volume(speed):
    r = np.where(speed < 0.19, np.sqrt(speed / 1.19e8), speed / 8000.0)
    return 4 / 3 * np.pi * r**3


def _state(nx, nz, per, dz, seed):
    """Every SD falls as many levels as it lies above the lowest."""
    rng = np.random.default_rng(seed)
    cell = np.repeat(np.arange(nx * nz, dtype=np.int32), per)
    n = len(cell)
    v = _volume(np.maximum(cell // nx * dz, 1e-3) * (1 + 1e-3 * rng.random(n)))
    xi = rng.integers(1, 1000, n).astype(np.int64)
    xi[rng.random(n) < 0.02] = 0
    p = rng.permutation(n)
    return xi[p], v[p], cell[p], np.full(n, 0.5 * dz)


# arrivals of the lowest cells: 1024 (the most that are merged), 1026, 1500, and
# 1200 in each of many; one piece of a grid (whose lowest level others lie below)
@pytest.mark.parametrize("nx,nz,per,base,steps", [(2, 3, 512, 0, 3), (2, 4, 342, 0, 3), (8, 6, 300, 0, 20),
                                                  (700, 4, 400, 0, 19), (5, 8, 300, 10, 20)])
def test_pile(env, nx, nz, per, base, steps):
    O, sdm, torch = env
    dz, nc = 0.3, nx * nz
    xi, v, cell, zeta = _state(nx, nz, per, dz, per)
    n = len(xi)
    run = sdm.Run(sdm.make_config("geometric", dv=1e3, n_cells=nc, seed=3, cell_base=base), n).set_attributes(xi, v, cell)
    sdm.sdm_set_heights(run.h, zeta, nx, dz)
    # the oracle's grid holds the levels below the piece, empty
    st = O.State(xi.copy(), v.copy(), cell + base, None, nc + base)
    P = O.params("geometric", dv=1e3, seed=3)
    for t in range(steps):
        run.sediment()
        O.sediment(P, st, nx, dz, zeta)
        gone = st.cell < base  # out of the piece
        gz, gc = sdm.sdm_get_heights(run.h)
        inside = ~gone
        assert np.array_equal(gc[inside], st.cell[inside]) and np.array_equal(gz[inside], zeta[inside]), f"step {t}"
        assert (gc[gone] < base).all()
        st.cell[gone] = -1
        run.step(1)
        O.step(P, st, t)
        x, w = run.attributes()
        assert np.array_equal(x, st.xi) and np.array_equal(w, st.v), f"step {t}"
    assert (st.cell >= 0).sum() < n
    run.close()


def test_time_of_a_pile(env):
    O, sdm, torch = env
    nx, nz, per, dz = 10, 64, 1000, 0.05
    xi, v, cell, zeta = _state(nx, nz, per, dz, 1)
    run = sdm.Run(sdm.make_config("geometric", dv=1e3, n_cells=nx * nz, seed=3), len(xi))
    times = []
    for _ in range(4):
        run.set_attributes(xi, v, cell)
        sdm.sdm_set_heights(run.h, zeta, nx, dz)
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        torch.cuda.synchronize()
        a.record()
        run.sediment()
        b.record()
        torch.cuda.synchronize()
        times.append(a.elapsed_time(b))
    assert run.info().largest_cell > 30000
    run.close()
    assert min(times) < 5.0, times  # ms: 120 merged by one block each, 0.15 sorted
