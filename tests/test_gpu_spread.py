"""Larger cells that hold few super-droplets in all (two launches per step over
buckets of equal key ranges), against the oracle bit for bit: sizes just above
the shared-memory classes and of a few buckets' remainder, cells whose live
super-droplets leave most buckets empty (pairs then cross many of them), odd
live counts, several runs in one batch, and the allocation-free step."""
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


def _state(n, live):
    rng = np.random.default_rng(n + live)
    xi = rng.integers(1, 10**9, n).astype(np.int64)
    xi[rng.permutation(n)[live:]] = 0
    return xi, 4 / 3 * np.pi * np.exp(rng.uniform(np.log(2e-6), np.log(1e-3), n)) ** 3


def _oracle(O, kernel, precision, xi, v, steps, dv, cell=None, n_cells=1):
    st = O.State(xi.copy(), v.copy(), np.zeros(len(xi), np.int32) if cell is None else cell, None, n_cells)
    O.run(O.params(kernel, precision, dv=dv, seed=5), st, 0, steps)
    return st


SIZES = [(4097, 4097), (4098, 4000), (4480, 4480), (4999, 3), (5000, 2), (5001, 1), (5002, 0), (8191, 60), (16384, 16383),
         (20000, 700), (131072, 131071)]


@pytest.mark.parametrize("kernel, precision, dv", [("golovin", "fp64", 1e2), ("geometric", "kfp32", 1e-2)])
@pytest.mark.parametrize("n, live", SIZES)
def test_one_cell(env, kernel, precision, dv, n, live):
    O, sdm, torch = env
    xi, v = _state(n, live)
    run = sdm.Run(sdm.make_config(kernel, precision, dv=dv, seed=5), n).set_attributes(xi, v, np.zeros(n, np.int32))
    run.step(2).step(3)
    x, w = run.attributes()
    run.close()
    st = _oracle(O, kernel, precision, xi, v, 5, dv)
    assert np.array_equal(x, st.xi) and np.array_equal(w, st.v)


@pytest.mark.parametrize("graph", [False, True])
def test_batch_of_cells(env, graph):
    O, sdm, torch = env
    runs, want = [], []
    for n, live in SIZES:
        xi, v = _state(n, live)
        runs.append(sdm.Run(sdm.make_config("golovin", dv=1e2, seed=5), n).set_attributes(xi, v, np.zeros(n, np.int32)))
        want.append(_oracle(O, "golovin", "fp64", xi, v, 7, 1e2))
    # a run of several cells, one of them in the shared-memory classes
    xi, v = _state(12000, 11000)
    cell = np.repeat(np.arange(3, dtype=np.int32), [5001, 300, 6699])
    runs.append(sdm.Run(sdm.make_config("golovin", dv=1e2, n_cells=3, seed=5), 12000).set_attributes(xi, v, cell))
    want.append(_oracle(O, "golovin", "fp64", xi, v, 7, 1e2, cell, 3))
    batch = sdm.Batch(runs, use_graph=graph, graph_steps=3)
    batch.step(6).step(1)
    for run, st in zip(runs, want):
        x, w = run.attributes()
        assert np.array_equal(x, st.xi) and np.array_equal(w, st.v)
    batch.close()


@pytest.mark.parametrize("n", [4098, 5002, 65536, 262144, 262146])
def test_noalloc(env, n):
    O, sdm, torch = env
    xi, v = _state(n, n - 7)
    cfg = sdm.make_config("golovin", dv=1e2, seed=5)
    x, w = torch.from_numpy(xi).cuda(), torch.from_numpy(v).cuda()
    for s in range(3):
        sdm.sdm_cell_step_noalloc(cfg, s, x, w, sdm.current_stream_handle())
    st = _oracle(O, "golovin", "fp64", xi, v, 3, 1e2)
    assert np.array_equal(x.cpu().numpy(), st.xi) and np.array_equal(w.cpu().numpy(), st.v)
