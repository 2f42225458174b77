"""One cell at the edges of the block kernel's sizes: the allocation-free step
and steps of a context (one launch each, and fused), against the oracle bit for
bit.  600 steps of 4096 super-droplets draw 1e6 sort words per bucket width, so
that words sharing their 32 key bits (0.2% of the steps) occur."""
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


def _state(n):
    rng = np.random.default_rng(n)
    xi = np.where(rng.random(n) < 0.3, 1000, rng.integers(1, 10**9, n)).astype(np.int64)
    xi[rng.random(n) < 0.1] = 0
    return xi, 4 / 3 * np.pi * np.exp(rng.uniform(np.log(2e-6), np.log(1e-3), n)) ** 3


def _oracle(O, kernel, xi, v, steps, dv):
    st = O.State(xi.copy(), v.copy(), np.zeros(len(xi), np.int32), None, 1)
    O.run(O.params(kernel, "fp64", dv=dv, seed=5), st, 0, steps)
    return st


@pytest.mark.parametrize("kernel", ["golovin", "geometric"])
@pytest.mark.parametrize("n", [2, 62, 64, 66, 128, 130, 256, 258, 512, 514, 1022, 1024, 1026, 2048, 2050, 4094, 4096,
                               4098])
def test_noalloc_sizes(env, kernel, n):
    O, sdm, torch = env
    xi, v = _state(n)
    cfg = sdm.make_config(kernel, dv=1e-3, seed=5)
    x, w = torch.from_numpy(xi).cuda(), torch.from_numpy(v).cuda()
    for s in range(3):
        sdm.sdm_cell_step_noalloc(cfg, s, x, w, sdm.current_stream_handle())
    st = _oracle(O, kernel, xi, v, 3, 1e-3)
    assert np.array_equal(x.cpu().numpy(), st.xi) and np.array_equal(w.cpu().numpy(), st.v)


@pytest.mark.parametrize("n, steps", [(513, 5), (1023, 5), (1024, 5), (1025, 5), (2047, 5), (2049, 5), (4096, 600)])
def test_block_cell_steps(env, n, steps):
    O, sdm, torch = env
    xi, v = _state(n)
    st = _oracle(O, "golovin", xi, v, steps, 1e2)
    for calls in ([steps], [1] * 3 + [steps - 3]):
        run = sdm.Run(sdm.make_config("golovin", dv=1e2, seed=5), n).set_attributes(xi, v, np.zeros(n, np.int32))
        for k in calls:
            run.step(k)
        x, w = run.attributes()
        run.close()
        assert np.array_equal(x, st.xi) and np.array_equal(w, st.v)
