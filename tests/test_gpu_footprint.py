"""sdm_footprint_bytes is an upper bound of what a run takes from its
allocator until after its steps, also for a run with one cell above the
record path's largest and others within it (both paths' scratch)."""
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


@pytest.mark.parametrize("sizes", [[(1 << 24) + 2, 1 << 24], [1 << 20] * 3, [4097] * 500, [240000], [239990, 8, 12],
                                   [60000, 60000, 20000, 5000], [100001]])
def test_bound(env, sizes):
    sdm, torch = env
    now, peak, live = [0], [0], {}

    def alloc(nbytes, stream, user):
        p = torch.cuda.caching_allocator_alloc(int(nbytes), torch.cuda.current_device(), stream or 0)
        live[p] = int(nbytes)
        now[0] += int(nbytes)
        peak[0] = max(peak[0], now[0])
        return p

    def free(ptr, nbytes, stream, user):
        if ptr:
            now[0] -= live.pop(ptr)
            torch.cuda.caching_allocator_delete(ptr)

    n, nc = sum(sizes), len(sizes)
    cfg = sdm.make_config("golovin", dv=1e8, n_cells=nc, seed=1)
    hooks = sdm.ALLOC_FN(alloc), sdm.FREE_FN(free)
    cfg.alloc, cfg.free = hooks
    run = sdm.Run(cfg, n, torch_memory=False)
    cell = torch.repeat_interleave(torch.arange(nc, dtype=torch.int32), torch.tensor(sizes)).cuda()
    run.set_attributes(torch.full((n,), 1000, dtype=torch.int64, device="cuda"),
                       torch.full((n,), 1e-14, dtype=torch.float64, device="cuda"), cell)
    run.step(2)
    torch.cuda.synchronize()
    bound = sdm.sdm_footprint_bytes(n, nc, max(sizes))
    run.close()
    assert peak[0] <= bound, (peak[0], bound)
