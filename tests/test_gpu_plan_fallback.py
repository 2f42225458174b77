"""Plans whose record rooms cannot be had: cells above mid_max_sd then take the
multi-pass path and the others the cluster path, with the oracle's results,
bit for bit.  The allocator hook refuses the rooms' size, as a full device
would.  (Here a plan holds several multi-pass cells, of several runs, with
their offsets into the shared scratch and their liveness bits; the
allocation-free step launches the same kernels for one cell.)"""
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


def _hooks(env, sizes):
    """Hooks that refuse the rooms of a plan with cells of these sizes (22.5 KB per
    1024 SDs or part of a cell), and anything larger."""
    O, sdm, torch = env
    refused, live = [], set()
    rooms = sum(-(-n // 1024) for n in sizes if n > 4096) * 1408 * 16

    def alloc(nbytes, stream, user):
        if nbytes >= rooms:
            refused.append(int(nbytes))
            return None
        p = torch.cuda.caching_allocator_alloc(int(nbytes), torch.cuda.current_device(), stream or 0)
        live.add(p)
        return p

    def free(ptr, nbytes, stream, user):
        if ptr:
            live.discard(ptr)
            torch.cuda.caching_allocator_delete(ptr)

    return sdm.ALLOC_FN(alloc), sdm.FREE_FN(free), refused, live


def _state(rng, sizes):
    cell = np.repeat(np.arange(len(sizes), dtype=np.int32), sizes)
    n = len(cell)
    xi = np.where(rng.random(n) < 0.3, 1000, rng.integers(1, 10**9, n)).astype(np.int64)
    xi[rng.random(n) < 0.05] = 0
    v = 4 / 3 * np.pi * np.exp(rng.uniform(np.log(2e-6), np.log(2e-3), n)) ** 3
    return xi, v, cell


def _same(env, run, kernel, precision, dv, seed, state, nc, steps):
    O, sdm, torch = env
    gx, gv = run.attributes()
    st = O.State(state[0].copy(), state[1].copy(), state[2].copy(), None, nc)
    O.run(O.params(kernel, precision, dv=dv, seed=seed), st, 0, steps)
    assert np.array_equal(gx, st.xi) and np.array_equal(gv, st.v)
    assert int((gx != state[0]).sum()) > 0


def _run(env, hooks, kernel, precision, dv, seed, state, nc):
    O, sdm, torch = env
    cfg = sdm.make_config(kernel, precision, dv=dv, n_cells=nc, seed=seed)
    cfg.alloc, cfg.free = hooks[:2]
    return sdm.Run(cfg, len(state[0]), torch_memory=False).set_attributes(*state)


@pytest.mark.parametrize("kernel,precision,dv", [("golovin", "fp64", 1e2), ("geometric", "kfp32", 1e1)])
def test_one_run(env, kernel, precision, dv):
    sizes = [16385, 70001, 4097, 700, 131074, 9000, 40001]
    state = _state(np.random.default_rng(3), sizes)
    hooks = _hooks(env, sizes)
    run = _run(env, hooks, kernel, precision, dv, 6, state, len(sizes))
    run.step(2).step(1)
    assert hooks[2], "the plan asked for no rooms"
    _same(env, run, kernel, precision, dv, 6, state, len(sizes), 3)
    run.close()
    env[2].cuda.synchronize()
    assert not hooks[3]


@pytest.mark.parametrize("graph", [False, True])
def test_batch(env, graph):
    O, sdm, torch = env
    rng = np.random.default_rng(4)
    layouts = ([100001, 300], [5001, 65537, 20000], [53000])
    hooks = _hooks(env, sum(layouts, []))
    members = []
    for i, sizes in enumerate(layouts):
        state = _state(rng, sizes)
        members.append((state, len(sizes), 20 + i, _run(env, hooks, "golovin", "fp64", 1e2, 20 + i, state, len(sizes))))
    batch = sdm.Batch([m[3] for m in members], use_graph=graph, graph_steps=2)
    batch.step(4)
    assert hooks[2]
    for state, nc, seed, run in members:
        _same(env, run, "golovin", "fp64", 1e2, seed, state, nc, 4)
    batch.close()
    for m in members:
        m[3].close()
    torch.cuda.synchronize()
    assert not hooks[3]
