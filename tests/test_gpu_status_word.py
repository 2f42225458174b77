"""A run's status word reaches the caller of every product that waits for its
result.

Bit 0: a bounded device wait gave up; bit 1: a sort bucket outgrew its room
and a cell was left unstepped (once in 1e30 steps by chance, so the word is
written here in place of the kernel: the run's record is the block that the
allocator hook handed out for it, and its words kernel, precision, n_cells
and status lie behind one another)."""
import numpy as np
import pytest

from paper_2103_17238_gb300 import inputs as I

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


def _run(env, n_cells, per_cell):
    """A context whose device blocks are tensors of this program."""
    sdm, torch = env
    blocks = {}

    def alloc(nbytes, stream, user):
        t = torch.empty(int(nbytes) + 256, dtype=torch.uint8, device="cuda")
        p = (t.data_ptr() + 255) & ~255
        blocks[p] = t[p - t.data_ptr():p - t.data_ptr() + int(nbytes)]
        return p

    def free(ptr, nbytes, stream, user):
        pass

    cfg = sdm.make_config("geometric", "fp64", dv=1e6, n_cells=n_cells, seed=5)
    hooks = sdm.ALLOC_FN(alloc), sdm.FREE_FN(free)
    cfg.alloc, cfg.free = hooks
    n = n_cells * per_cell
    h = sdm.sdm_create(cfg, n, sdm.current_stream_handle())
    own = list(blocks.values())  # (a later block is the upload's, with a copy of the record)
    rng = np.random.default_rng(3)
    xi = rng.integers(1, 10**6, n).astype(np.int64)
    v = 4 / 3 * np.pi * np.exp(rng.uniform(np.log(3e-6), np.log(3e-4), n)) ** 3
    sdm.sdm_set_attributes(h, xi, v, np.repeat(np.arange(n_cells, dtype=np.int32), per_cell))
    torch.cuda.synchronize()
    status = None
    for t in own:
        if t.numel() > 512 or t.numel() % 4:
            continue
        w = t.view(torch.int32)
        at = [i for i in range(w.numel() - 3) if w[i:i + 4].tolist() == [1, 0, n_cells, 0]]
        if at:
            assert status is None and len(at) == 1
            status = w[at[0] + 3:at[0] + 4]
    assert status is not None
    return h, status, (hooks, blocks)


def _error(sdm, call):
    """(status, message) of the call's error; nothing keeps its frames alive."""
    try:
        call()
    except sdm.SdmError as err:
        return err.status, str(err)
    return sdm.SDM_OK, ""


@pytest.mark.parametrize("n_cells,per_cell", [(37, 200), (37, 9000), (1, 3000)])
@pytest.mark.parametrize("bit,name", [(1, "SDM_ETIMEOUT"), (2, "SDM_ESTATE")])
def test_products_report_the_status(env, n_cells, per_cell, bit, name):
    sdm, torch = env
    h, status, keep = _run(env, n_cells, per_cell)
    calls = {
        "spectrum": lambda: sdm.sdm_spectrum(h, I.R_EDGES),
        "spectrum of many bins": lambda: sdm.sdm_spectrum(h, np.geomspace(1e-6, 1e-2, 60)),
        "cells' spectra": lambda: sdm.sdm_spectrum(h, I.R_EDGES, per_cell=True),
        "diagnostics": lambda: sdm.sdm_diagnostics(h),
        "attributes": lambda: sdm.sdm_get_attributes(h),
    }
    for call in calls.values():
        call()
    status.fill_(bit)
    torch.cuda.synchronize()
    for what, call in calls.items():
        assert _error(sdm, call)[0] == getattr(sdm, name), what
    status.fill_(0)
    torch.cuda.synchronize()
    for call in calls.values():
        call()
    sdm.sdm_destroy(h)
    torch.cuda.synchronize()
    keep[1].clear()  # (the hooks' closures hold one another)
