"""The precipitated water of a sedimentation step is the exactly rounded sum
of xi v over the SDs that fell through the bottom: it does not depend on the
path that took the step, so a run resumed from a checkpoint gives the same
bits as the run that went on."""
from fractions import Fraction

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


def _state(nx, nz, per, seed, r_lo, r_hi, dz):
    rng = np.random.default_rng(seed)
    nc = nx * nz
    cell = np.repeat(np.arange(nc, dtype=np.int32), per)
    n = len(cell)
    xi = rng.integers(1, 10**9, n).astype(np.int64)
    xi[rng.random(n) < 0.03] = 0
    xi[rng.random(n) < 0.01] = 2**62 + 3
    v = 4 / 3 * np.pi * np.exp(rng.uniform(np.log(r_lo), np.log(r_hi), n)) ** 3
    zeta = rng.random(n) * dz * 0.999
    return xi, v, cell, zeta


def _exact(xi, v, gone):
    return float(sum((Fraction(int(x)) * Fraction(float(w)) for x, w in zip(xi[gone], v[gone])), Fraction(0)))


# (cells few enough that heavy rain changes the path; above a warp's largest
# cell; many cells)
@pytest.mark.parametrize("nx,nz,per,r_lo,r_hi,dz", [(8, 4, 300, 1e-4, 2e-3, 4.0), (3, 3, 700, 2e-6, 3e-3, 2.0),
                                                    (2, 2, 3000, 1e-4, 2e-3, 5.0), (160, 5, 40, 1e-5, 2e-3, 3.0),
                                                    (4, 1, 64, 1e-4, 2e-3, 1.0), (500, 1, 900, 1e-4, 2e-3, 0.5)])
def test_resumed_run_and_exact_sum(env, nx, nz, per, r_lo, r_hi, dz):
    sdm, torch = env
    nc = nx * nz
    xi, v, cell, zeta = _state(nx, nz, per, 5, r_lo, r_hi, dz)
    run = sdm.Run(sdm.make_config("geometric", dv=1.0, n_cells=nc, seed=9), len(xi)).set_attributes(xi, v, cell)
    sdm.sdm_set_heights(run.h, zeta, nx, dz)
    fell = 0
    for step in range(4):
        z0, c0 = sdm.sdm_get_heights(run.h)
        x0, v0 = run.attributes()
        got = run.sediment()
        other = sdm.Run(sdm.make_config("geometric", dv=1.0, n_cells=nc, seed=9, step0=0), len(xi))
        other.set_attributes(x0, v0, c0.astype(np.int32))
        sdm.sdm_set_heights(other.h, z0, nx, dz)
        resumed = other.sediment()
        c1 = sdm.sdm_get_heights(run.h)[1]
        gone = (c0 >= 0) & (c1 < 0) & (x0 > 0)
        fell += int(gone.sum())
        want = _exact(x0, v0, gone)
        assert got == want, (step, got, want, int(gone.sum()))
        assert resumed == got
        assert np.array_equal(sdm.sdm_get_heights(other.h)[1], c1)
        other.close()
    assert fell > 100
    run.close()


def test_negative_and_cancelling(env):
    """Volumes of both signs (over-evaporated drops fall as drops of |v|) and
    sums that cancel to zero."""
    sdm, torch = env
    n = 600
    rng = np.random.default_rng(8)
    xi = rng.integers(1, 10**9, n).astype(np.int64)
    v = 4 / 3 * np.pi * np.exp(rng.uniform(np.log(1e-5), np.log(1e-4), n)) ** 3
    run = sdm.Run(sdm.make_config("geometric", dt=300.0, dv=1.0, n_cells=2, seed=2), n)
    run.set_attributes(xi, v, np.repeat(np.arange(2, dtype=np.int32), n // 2))
    run.condense(np.full(2, 1e-10), np.full(2, -0.2), 1e-9, want_condensed=False)
    w = run.attributes()[1]
    assert (w < 0).any() and (w > 0).any()
    sdm.sdm_set_heights(run.h, np.zeros(n), 1, 1e-9)
    got = run.sediment()
    gone = sdm.sdm_get_heights(run.h)[1] < 0
    assert gone.sum() > n // 2
    assert got == _exact(xi, w, gone)
    assert run.sediment() == _exact(xi, w, ~gone & (sdm.sdm_get_heights(run.h)[1] < 0))
    run.close()
