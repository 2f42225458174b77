"""A run of larger cells that sediments: its launch plan is made anew at every
step, but not the plan's rooms, which go from one plan to the next (with some
to spare once a layout has outgrown them); a layout that needs none gives them
back, and so does the run's end."""
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


# record path; bucketed path
@pytest.mark.parametrize("sizes", [[80000, 90001, 100000, 6000], [20000, 30001, 40000, 6000]])
def test_rooms_stay(env, sizes):
    O, sdm, torch = env
    large, live = [], {}

    def alloc(nbytes, stream, user):
        p = torch.cuda.caching_allocator_alloc(int(nbytes), torch.cuda.current_device(), stream or 0)
        live[p] = int(nbytes)
        if nbytes > 1 << 20:
            large.append(int(nbytes))
        return p

    def free(ptr, nbytes, stream, user):
        if ptr:
            live.pop(ptr)
            torch.cuda.caching_allocator_delete(ptr)

    rng = np.random.default_rng(3)
    nc, dz = len(sizes), 10.0
    cell = np.repeat(np.arange(nc, dtype=np.int32), sizes)
    n = len(cell)
    xi = rng.integers(1, 10**6, n).astype(np.int64)
    v = 4 / 3 * np.pi * np.exp(rng.uniform(np.log(1e-5), np.log(1e-4), n)) ** 3
    zeta = rng.random(n) * dz
    cfg = sdm.make_config("geometric", dv=1e3, n_cells=nc, seed=4)
    hooks = sdm.ALLOC_FN(alloc), sdm.FREE_FN(free)
    cfg.alloc, cfg.free = hooks
    run = sdm.Run(cfg, n, torch_memory=False)
    dev = [torch.as_tensor(a, device="cuda") for a in (xi, v, cell, zeta)]
    run.set_attributes(*dev[:3])
    sdm.sdm_set_heights(run.h, dev[3], 1, dz)
    st = O.State(xi.copy(), v.copy(), cell.copy(), None, nc)
    P = O.params("geometric", dv=1e3, seed=4)
    for t in range(8):
        run.step(1)
        if t == 0:
            del large[:]
        run.sediment()
        O.step(P, st, t)
        O.sediment(P, st, 1, dz, zeta)
    run.step(1)
    O.step(P, st, 8)
    x, w = run.attributes()
    assert np.array_equal(x, st.xi) and np.array_equal(w, st.v)
    torch.cuda.synchronize()
    staging = 16 * n  # sdm_get_attributes' own
    assert len([b for b in large if b != staging]) <= 1  # eight plans, outgrown once at most
    held = sum(live.values())
    assert run.info().device_bytes <= held
    small = np.zeros(n, np.int32)
    small[:] = np.arange(n) % nc
    run.set_attributes(*(torch.as_tensor(a[:4000], device="cuda") for a in (xi, v, small))).step(1)
    torch.cuda.synchronize()
    assert sum(live.values()) < held - (1 << 20)
    run.close()
    torch.cuda.synchronize()
    assert not live
