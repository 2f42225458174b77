"""The sedimentation step by cells (each new cell merged from its stayers and
its arrivals) against the oracle, at the sizes where it can go wrong: every SD
of a cell falling at once (up to, and beyond, the 512 arrivals sorted in shared
memory; few cells go over to the sort then, many do not), cells about 1024 slots (above it all SDs are sorted instead, and the
layout passes from one path to the other), over 65,536 cells (offsets over
block totals), and a piece of a grid."""
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


def _run(env, sizes, nx, dt, r_lo, r_hi, steps, seed, levels=None):
    O, sdm, torch = env
    rng = np.random.default_rng(seed)
    n_cells, dz = len(sizes), 10.0
    cell = np.repeat(np.arange(n_cells, dtype=np.int32), sizes)
    n = len(cell)
    r = np.exp(rng.uniform(np.log(r_lo), np.log(r_hi), n))
    if levels is not None:  # every SD as many times larger as it shall fall levels
        r *= np.maximum(levels[cell], 0.01)
    v = 4 / 3 * np.pi * r**3
    xi = rng.integers(1, 10**6, n).astype(np.int64)
    xi[rng.random(n) < 0.02] = 0
    zeta = rng.uniform(0.0, dz, n)
    perm = rng.permutation(n)
    xi, v, cell, zeta = xi[perm], v[perm], cell[perm], zeta[perm]
    run = sdm.Run(sdm.make_config("geometric", dt=dt, dv=1e6, n_cells=n_cells, seed=3), n)
    run.set_attributes(xi, v, cell)
    sdm.sdm_set_heights(run.h, zeta, nx, dz)
    st = O.State(xi.copy(), v.copy(), cell.copy(), None, n_cells)
    P = O.params("geometric", dt=dt, dv=1e6, seed=3)
    moved = 0
    for t in range(steps):
        before = st.cell.copy()
        got, want = run.sediment(), O.sediment(P, st, nx, dz, zeta)
        assert abs(got - want) <= 1e-12 * want
        moved += int((st.cell != before).sum())
        gz, gc = sdm.sdm_get_heights(run.h)
        assert np.array_equal(gc, st.cell), f"cells differ after step {t}"
        inside = st.cell >= 0
        assert np.array_equal(gz[inside], zeta[inside]), f"heights differ after step {t}"
        run.step(1)
        O.step(P, st, t)
        x, w = run.attributes()
        assert np.array_equal(x, st.xi) and np.array_equal(w, st.v), f"state differs after step {t}"
    assert moved > 0
    run.close()


@pytest.mark.parametrize("per", [31, 500, 512, 530, 900])
def test_whole_cells_fall(env, per):
    _run(env, [per] * 5, 1, 10.0, 1.2e-4, 1.24e-4, 4, per)  # about 9.7 m per step of levels of 10 m


@pytest.mark.parametrize("sizes", [(1023, 1, 1024, 2), (1024, 1025, 3, 0), (1000, 900, 100, 1024)])
def test_about_the_largest_cell(env, sizes):
    _run(env, list(sizes) * 3, 4, 2.0, 1e-5, 1e-3, 4, sum(sizes))


def test_many_cells(env):
    _run(env, list(np.random.default_rng(1).integers(0, 4, 70000)), 100, 5.0, 1e-5, 1e-3, 2, 9)


@pytest.mark.parametrize("per", [300, 700, 1000])
def test_cells_pile_up(env, per):
    # four levels fall into the lowest: 4 per arrivals there (2048 are one run of the block's sort)
    _run(env, [per, per, per - 1, per, per + 1], 1, 10.0, 1.24e-4, 1.26e-4, 2, per, levels=np.arange(5))


@pytest.mark.parametrize("per", [257, 500, 1000])
def test_whole_cells_fall_among_many(env, per):
    _run(env, [per] * 5 + [2] * 640, 1, 10.0, 1.2e-4, 1.24e-4, 4, per)


@pytest.mark.parametrize("per", [200, 700])
def test_cells_pile_up_among_many(env, per):
    levels = np.concatenate([np.arange(5), np.zeros(640)])
    _run(env, [per, per, per - 1, per, per + 1] + [2] * 640, 1, 10.0, 1.24e-4, 1.26e-4, 2, per, levels=levels)
