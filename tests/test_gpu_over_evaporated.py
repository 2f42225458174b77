"""Sums over super-droplets whose volume an evaporating condensation step has
left below zero.

The step adds a binary32 change to the binary64 volume, so where a drop
shrinks to a floor some 150 times below its radius, the change's rounding
(about 2^-22 of the volume) exceeds what is left, and v can end slightly
negative.  The oracle's sums take such an SD with its sign: sum(xi v) counts
it negative, and the spectrum puts xi v into the bin of the radius of |v|."""
import math
from fractions import Fraction

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

G, S, R_MIN, DT = 1.0e-10, -0.2, 1.0e-9, 300.0


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


def _evaporated(env, sizes):
    O, sdm, torch = env
    rng = np.random.default_rng(41)
    cell = np.repeat(np.arange(len(sizes), dtype=np.int32), sizes)
    n = len(cell)
    xi = rng.integers(1, 10**9, n).astype(np.int64)
    xi[rng.random(n) < 0.05] = 0
    xi[rng.random(n) < 0.02] = 2**60 + 12345
    v = 4 / 3 * np.pi * np.exp(rng.uniform(np.log(1e-5), np.log(1e-4), n)) ** 3
    nc = len(sizes)
    run = sdm.Run(sdm.make_config("geometric", dt=DT, dv=1.0, n_cells=nc, seed=2), n).set_attributes(xi, v, cell)
    run.condense(np.full(nc, G), np.full(nc, S), R_MIN, want_condensed=False)
    st = O.State(xi.copy(), v.copy(), cell.copy(), None, nc)
    P = O.params("geometric", dt=DT, dv=1.0, seed=2)
    O.condense(P, st, np.full(nc, G), np.full(nc, S), R_MIN)
    assert np.array_equal(run.attributes()[1], st.v)
    assert ((st.v < 0) & (st.xi > 0)).mean() > 0.2
    return run, st, P


def _terms(xi, v):
    return [Fraction(int(x)) * Fraction(float(w)) for x, w in zip(xi, v)]


@pytest.mark.parametrize("sizes", [[64, 1000, 3, 256], [9000, 1]])
def test_sum_of_water(env, sizes):
    """Within the rounding of one binary64 addition per SD of either sign."""
    run, st, _ = _evaporated(env, sizes)
    t = _terms(st.xi, st.v)
    want, mag = sum(t), sum(abs(x) for x in t)
    d = run.diagnostics()
    assert d["live_sd"] == int((st.xi > 0).sum()) and d["sum_xi"] == sum(int(x) for x in st.xi)
    assert abs(Fraction(d["sum_xi_v"]) - want) <= len(t) * mag / 2**53
    run.close()


@pytest.mark.parametrize("per_cell", [False, True])
@pytest.mark.parametrize("bins", [1, 31, 40])
@pytest.mark.parametrize("sizes", [[64, 1000, 3, 256], [9000, 1], [2500]])
def test_spectrum(env, sizes, bins, per_cell):
    O, sdm, torch = env
    run, st, P = _evaporated(env, sizes)
    edges = np.exp(np.linspace(np.log(1e-8), np.log(2e-6), bins + 1))
    got = run.spectrum(edges, per_cell=per_cell)
    want = O.spectrum(P, st, edges, per_cell=per_cell)
    pos = O.State(st.xi, np.abs(st.v), st.cell, None, st.n_cells)
    mag = O.spectrum(P, pos, edges, per_cell=per_cell)
    assert mag.max() > 0 and ((want < 0).any() or bins == 1)
    assert np.all(np.abs(got - want) <= 2 * (len(st.xi) + 4) * 2.0**-53 * mag)
    run.close()
