"""What a step leaves behind when a device wait gives up, on a build of the
library in which some waits give up at once (tests/give_up.cu: the copies they
wait for still arrive, and the kernel waits for them before it leaves, so
nothing is out of range and the device stays usable).

Record path: the SDs of a bucket that gave up stay as they were, with the
partners that a pair across its ends would have had; every other pair is
stepped as the oracle steps it; the call that reads the state reports
SDM_ETIMEOUT; and the next step finds its counts in order.

Allocation-free step: a call takes nothing from what its array held before, so
calls that went wrong (overlapping ones, a launch that failed) spoil no later one;
and what a kernel reports, the next call says, once."""
import gc
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env(tmp_path_factory):
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from oracle import oracle as O
    from paper_2103_17238_gb300 import build as B
    from paper_2103_17238_gb300 import sdm

    O.build()
    path = str(tmp_path_factory.mktemp("give_up") / "libsdm_give_up.so")
    here = os.path.dirname(os.path.abspath(__file__))
    subprocess.run([B.nvcc(), *B.NVCC_FLAGS, os.path.join(here, "give_up.cu"), "-o", path], check=True)
    torch.cuda.set_device(0)
    gc.collect()  # runs that earlier tests left go with the library that made them
    before, sdm._lib = sdm._lib, None
    sdm.load(path)
    yield O, sdm, torch
    gc.collect()
    sdm._lib = before


def _error(sdm, call):
    """(status, message) of the call's error; nothing keeps its frames alive."""
    try:
        call()
    except sdm.SdmError as err:
        return err.status, str(err)
    return sdm.SDM_OK, ""


def _buckets_that_gave_up(O, seed, cell, s, ranks, nb):
    b = np.array([(O.sort_key(seed, int(r), cell, s) * nb) >> 64 for r in ranks])
    assert np.all(np.diff(b) >= 0)
    return b % 3 == 1


# several cells and cells that share a launch without and with the launch that scans the counts
@pytest.mark.parametrize("sizes,steps", [([200001, 3, 40002, 5000], 3), ([(1 << 21) + 4098], 1)])
def test_record_path(env, sizes, steps):
    O, sdm, torch = env
    rng = np.random.default_rng(23)
    nc, seed, dv = len(sizes), 11, 1e-1
    cell = np.repeat(np.arange(nc, dtype=np.int32), sizes)
    n = len(cell)
    xi = rng.integers(1, 10**9, n).astype(np.int64)
    xi[rng.random(n) < 0.05] = 0
    v = 4 / 3 * np.pi * np.exp(rng.uniform(np.log(2e-6), np.log(2e-3), n)) ** 3
    run = sdm.Run(sdm.make_config("golovin", dv=dv, n_cells=nc, seed=seed), n).set_attributes(xi, v, cell)
    st = O.State(xi.copy(), v.copy(), cell.copy(), None, nc)
    P = O.params("golovin", dv=dv, seed=seed)
    dx = torch.empty(n, dtype=torch.int64, device="cuda")
    dw = torch.empty(n, dtype=torch.float64, device="cuda")
    for s in range(steps):
        x0, v0 = st.xi.copy(), st.v.copy()
        O.step(P, st, s)
        stepped = (st.xi != x0) | (st.v != v0)
        kept = np.zeros(n, bool)
        for c, size in enumerate(sizes):
            if size <= 4096:
                continue
            first = int(np.searchsorted(cell, c))
            perm = O.permutation(seed, c, s, x0[first:first + size])
            out = _buckets_that_gave_up(O, seed, c, s, perm, -(-size // 1024))
            pairs = perm[:len(perm) // 2 * 2].reshape(-1, 2)
            kept[first + pairs[out[:len(perm) // 2 * 2].reshape(-1, 2).any(axis=1)].ravel()] = True
        st.xi[kept], st.v[kept] = x0[kept], v0[kept]
        assert (stepped & kept).sum() > 1000 and (stepped & ~kept).sum() > 1000
        run.step(1)
        sdm.sdm_get_attributes(run.h, xi=dx, volume=dw)
        torch.cuda.synchronize()
        bad = np.nonzero((dx.cpu().numpy() != st.xi) | (dw.cpu().numpy() != st.v))[0]
        assert bad.size == 0, f"step {s}: {bad.size} SDs differ, first {bad[:5]} (cells {cell[bad[:5]]})"
    assert _error(sdm, run.attributes)[0] == sdm.SDM_ETIMEOUT
    run.close()


@pytest.mark.parametrize("fill", [0xFF, 0x01])
@pytest.mark.parametrize("n", [4096, 4098, 20000, 131072, 1 << 18, (1 << 18) + 2])
def test_noalloc_takes_nothing_from_before(env, n, fill):
    O, sdm, torch = env
    rng = np.random.default_rng(n)
    xi = rng.integers(1, 10**9, n).astype(np.int64)
    xi[rng.random(n) < 0.05] = 0
    v = 4 / 3 * np.pi * np.exp(rng.uniform(np.log(2e-6), np.log(2e-3), n)) ** 3
    dx, dw = torch.from_numpy(xi).cuda(), torch.from_numpy(v).cuda()
    cfg = sdm.make_config("golovin", dv=1e-1, n_cells=1, seed=3)
    stream = sdm.current_stream_handle()
    warm = torch.ones(64, dtype=torch.int64, device="cuda"), torch.full((64,), 1e-15, dtype=torch.float64, device="cuda")
    sdm.sdm_cell_step_noalloc(cfg, 0, *warm, stream)
    torch.cuda.synchronize()
    st = O.State(xi.copy(), v.copy(), np.zeros(n, np.int32), None, 1)
    P = O.params("golovin", dv=1e-1, seed=3)
    for s in range(2):
        assert sdm.load().give_up_fill_noalloc(fill) == 0
        sdm.sdm_cell_step_noalloc(cfg, s, dx, dw, stream)
        torch.cuda.synchronize()
        O.step(P, st, s)
        assert np.array_equal(dx.cpu().numpy(), st.xi) and np.array_equal(dw.cpu().numpy(), st.v)
    assert int((st.xi != xi).sum()) > 0


@pytest.mark.parametrize("n", [64, 5000, 1 << 19])
@pytest.mark.parametrize("which,name", [(0, "SDM_ETIMEOUT"), (1, "SDM_ESTATE")])
def test_noalloc_reports(env, which, name, n):
    O, sdm, torch = env
    dx = torch.full((n,), 1000, dtype=torch.int64, device="cuda")
    dw = torch.full((n,), 1e-9, dtype=torch.float64, device="cuda")
    cfg = sdm.make_config("golovin", dv=1e-3, n_cells=1, seed=3)
    stream = sdm.current_stream_handle()
    sdm.sdm_cell_step_noalloc(cfg, 0, dx, dw, stream)
    torch.cuda.synchronize()
    x0, w0 = dx.clone(), dw.clone()
    assert sdm.load().give_up_report(which) == 0
    status, message = _error(sdm, lambda: sdm.sdm_cell_step_noalloc(cfg, 1, dx, dw, stream))
    assert status == getattr(sdm, name) and "earlier call" in message
    torch.cuda.synchronize()
    assert torch.equal(dx, x0) and torch.equal(dw, w0)
    sdm.sdm_cell_step_noalloc(cfg, 1, dx, dw, stream)
    sdm.sdm_cell_step_noalloc(cfg, 2, dx, dw, stream)
    torch.cuda.synchronize()
    assert not torch.equal(dx, x0)
