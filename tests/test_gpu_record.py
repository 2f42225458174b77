"""The record path of larger cells (plans of more than 240,000 SDs in cells
above 4096: records of 16 bytes scattered into buckets, ordered and paired
there) against the oracle, bit for bit, at the sizes where it can go wrong:
about chunks of 4096 and buckets of 1024, odd sizes, cells with few SDs alive
(empty buckets between two that share a pair), a cell of thousands of buckets
(where key bits tie), more than one group of cells, and the other paths' results."""
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


def _state(rng, sizes, dead=0.05):
    cell = np.repeat(np.arange(len(sizes), dtype=np.int32), sizes)
    n = len(cell)
    xi = np.where(rng.random(n) < 0.3, 1000, rng.integers(1, 10**9, n)).astype(np.int64)
    xi[rng.random(n) < dead] = 0
    v = 4 / 3 * np.pi * np.exp(rng.uniform(np.log(2e-6), np.log(2e-3), n)) ** 3
    return xi, v, cell


def _check(env, kernel, precision, dv, xi, v, cell, n_cells, chunks, seed=13):
    O, sdm, torch = env
    run = sdm.Run(sdm.make_config(kernel, precision, dv=dv, n_cells=n_cells, seed=seed), len(xi))
    run.set_attributes(xi, v, cell)
    for k in chunks:
        run.step(k)
    gx, gv = run.attributes()
    run.close()
    st = O.State(xi.copy(), v.copy(), cell.copy(), None, n_cells)
    O.run(O.params(kernel, precision, dv=dv, seed=seed), st, 0, sum(chunks))
    bad = np.nonzero(gx != st.xi)[0]
    assert bad.size == 0, f"{bad.size} multiplicities differ, first at SD {bad[0]} (cell {cell[bad[0]]})"
    assert np.array_equal(gv, st.v)
    assert int((gx != xi).sum()) > 0


SIZES = [4097, 4098, 5119, 5121, 8191, 8193, 16385, 20001, 65536, 70001, 131073, 3, 700]


@pytest.mark.parametrize("kernel,precision,dv", [("golovin", "fp64", 1e2), ("geometric", "fp64", 1e-3),
                                                 ("long", "fp64", 1e1), ("geometric", "kfp32", 1e1),
                                                 ("golovin", "fp64", 1e-4)])
def test_sizes(env, kernel, precision, dv):
    rng = np.random.default_rng(17)
    _check(env, kernel, precision, dv, *_state(rng, SIZES), len(SIZES), [2, 1])


@pytest.mark.parametrize("alive", [(11, 7, 2, 1), (500, 301, 40, 0)])
def test_mostly_dead(env, alive):
    rng = np.random.default_rng(5)
    sizes = [150000, 120000, 30000, 5000]
    xi, v, cell = _state(rng, sizes, dead=0.0)
    for c, k in enumerate(alive):
        idx = np.nonzero(cell == c)[0]
        xi[np.setdiff1d(idx, rng.choice(idx, k, replace=False))] = 0
    _check(env, "golovin", "fp64", 1e-7, xi, v, cell, 4, [1, 2])


def test_thousands_of_buckets(env):
    rng = np.random.default_rng(6)
    _check(env, "golovin", "fp64", 1e4, *_state(rng, [4194305]), 1, [2])


def test_groups_of_cells(env):
    """17 boxes of 2^20 (two groups) equal the same boxes each stepped by itself,
    and the first equals the allocation-free step (multi-pass)."""
    O, sdm, torch = env
    n, m = 1 << 20, 17
    rng = np.random.default_rng(8)
    xi, v, cell = _state(rng, [n])
    dx, dw, dc = (torch.as_tensor(a, device="cuda") for a in (xi, v, cell))
    cfg = [sdm.make_config("golovin", dv=1e4, n_cells=1, seed=40 + i) for i in range(m)]
    runs = [sdm.Run(c, n).set_attributes(dx, dw, dc) for c in cfg]
    batch = sdm.Batch(runs, use_graph=True, graph_steps=2)
    batch.step(2)
    for i in (0, 7, 15, 16):
        alone = sdm.Run(cfg[i], n).set_attributes(dx, dw, dc)
        alone.step(2)
        a, b = runs[i].attributes(), alone.attributes()
        assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1]), f"box {i}"
        alone.close()
    stream = sdm.current_stream_handle()
    for s in range(2):
        sdm.sdm_cell_step_noalloc(cfg[0], s, dx, dw, stream)
    torch.cuda.synchronize()
    a = runs[0].attributes()
    assert np.array_equal(a[0], dx.cpu().numpy()) and np.array_equal(a[1], dw.cpu().numpy())
    assert int((a[0] != xi).sum()) > 0
