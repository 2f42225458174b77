"""Device buffers for the condensed water at any address: one that does not lie
on eight bytes receives the same values as an aligned one (a copy writes it)."""
import ctypes

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


@pytest.mark.parametrize("offset", [8, 4, 1])
@pytest.mark.parametrize("sizes", [[3, 256, 0, 700], [5000, 2]])
def test_address(env, sizes, offset):
    sdm, torch = env
    rng = np.random.default_rng(2)
    nc = len(sizes)
    cell = np.repeat(np.arange(nc, dtype=np.int32), sizes)
    n = len(cell)
    xi = rng.integers(1, 10**9, n).astype(np.int64)
    v = 4 / 3 * np.pi * np.exp(rng.uniform(np.log(1e-6), np.log(1e-3), n)) ** 3
    G, s = np.full(nc, 1e-10), rng.uniform(-0.01, 0.01, nc)
    got = []
    for at in (0, offset):
        run = sdm.Run(sdm.make_config("geometric", dv=1.0, n_cells=nc, seed=1), n).set_attributes(xi, v, cell)
        buf = torch.full((8 * nc + 64,), 0x5A, dtype=torch.uint8, device="cuda")
        assert buf.data_ptr() % 16 == 0
        st = sdm.load().sdm_condensation_step(run.h, G.ctypes.data_as(ctypes.c_void_p), s.ctypes.data_as(ctypes.c_void_p),
                                              1e-6, ctypes.c_void_p(buf.data_ptr() + at), 1)
        assert st == sdm.SDM_OK
        torch.cuda.synchronize()
        b = buf.cpu().numpy()
        assert (b[:at] == 0x5A).all() and (b[at + 8 * nc:] == 0x5A).all()
        got.append(b[at:at + 8 * nc].tobytes())
        run.close()
    assert got[0] == got[1]
    assert np.frombuffer(got[0]).any()
