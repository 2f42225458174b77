"""The condensation step in a captured graph: with a field that the context
has had before, the call is a launch and nothing else, so a program can
capture it and replay it; the volumes stay the oracle's, bit for bit."""
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


@pytest.mark.parametrize("water", [False, True])
@pytest.mark.parametrize("sizes", [[0, 1, 2, 63, 256, 700, 1024], [5, 0, 4097, 300]])
def test_replayed(env, sizes, water):
    O, sdm, torch = env
    rng = np.random.default_rng(12)
    nc = len(sizes)
    cell = np.repeat(np.arange(nc, dtype=np.int32), sizes)
    n = len(cell)
    xi = rng.integers(1, 10**9, n).astype(np.int64)
    v = 4 / 3 * np.pi * np.exp(rng.uniform(np.log(1e-6), np.log(1e-3), n)) ** 3
    G, s = np.full(nc, 1e-10), rng.uniform(-0.01, 0.01, nc)
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        run = sdm.Run(sdm.make_config("geometric", dv=1.0, n_cells=nc, seed=1), n).set_attributes(xi, v, cell)
        out = torch.zeros(nc, dtype=torch.float64, device="cuda") if water else None

        def step(f=s):
            sdm.sdm_condensation_step(run.h, G, f, 1e-6, want_condensed=water, n_cells=nc, out=out)

        step()
    stream.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        step()
    with torch.cuda.stream(stream):
        for _ in range(5):
            graph.replay()
        step(-s)  # another field behind the replays, more often than it has staging
        for _ in range(5):
            step(0.5 * s)
            step(s)
    stream.synchronize()
    st = O.State(xi.copy(), v.copy(), cell.copy(), None, nc)
    P = O.params("geometric", dv=1.0, seed=1)
    for f in [s] * 6 + [-s] + [0.5 * s, s] * 5:
        O.condense(P, st, G, f, 1e-6)
    assert np.array_equal(run.attributes()[1], st.v)
    run.close()
