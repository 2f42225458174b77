"""The work a user of this library has it do, as cases that can be timed and checked.

Every case goes through the Python binding (``paper_2103_17238_gb300.sdm``), as a program does:
a run or a batch that it keeps, attributes from its own arrays, steps, and the state and
products read back.  A pass that advances a run starts by setting the run's attributes, so
that every pass does the same amount of work; the two kinds that cannot (a batch keeps its
layout, the allocation-free step works on the caller's arrays) go on from where they are.

Kinds:
  cell      one allocation-free step of one cell in the caller's arrays: the smallest call
  box       one Golovin box, the paper's worked example: attributes in, n steps in one call,
            spectrum and attributes out (host arrays or device tensors)
  grid      a grid of cells: attributes in, n steps in one call or in n calls, spectrum (total
            or per cell) and attributes out
  coupled   a grid stepped by coalescence, condensation and sedimentation in turn
  batch     several boxes and grids in one batch, graph-replayed: an ensemble, or what a
            serving loop has running
  condense  condensation alone on a grid, an updraught's step and a downdraught's
  products  spectra and conservation sums of a standing state
  restore   a checkpoint in super-droplet order (cells in no order, as sedimentation leaves
            them) loaded with its positions and read back
"""
import math

import numpy as np
import torch

from paper_2103_17238_gb300 import inputs, sdm

DT_CHOICES = (0.5, 1.0, 2.0)
R_MIN = 1e-6


# ------------------------------------------------------------------ the cases
def listed():
    return [
        # a host model's own cell, one call per step: launches and latency
        dict(name="cell-1000", kind="cell", n_sd=1000, kernel="golovin", precision="fp64", dt=0.05),
        # the paper's worked example, small: host arrays in and out, many steps in one call
        dict(name="box-4096", kind="box", n_sd=4096, steps=200, host=True, precision="fp64"),
        # the paper's Golovin setting: one box of 2^17, an output interval
        dict(name="box-131072", kind="box", n_sd=131072, steps=60, host=False, precision="fp64"),
        # the 128 x 128 x 256 grid with a developed spectrum, an output interval in one call
        dict(name="grid-256", kind="grid", nx=128, nz=128, per_cell=256, ragged=False, developed=True, steps=30,
             one_call=True, kernel="geometric", precision="fp64", cell_spectrum=False),
        # cells of many sizes, Long's efficiency, binary32 kernel, one call per step
        # (something else happens between the steps), a spectrum of every cell
        dict(name="grid-ragged-long", kind="grid", nx=67, nz=61, per_cell=211, ragged=True, developed=True, steps=6,
             one_call=False, kernel="long", precision="kfp32", cell_spectrum=True),
        # the grid as 128 columns of 128 levels with all three dynamics
        dict(name="coupled-256", kind="coupled", nx=128, nz=128, per_cell=256, ragged=False, steps=6,
             kernel="geometric", precision="fp64"),
        # an ensemble of boxes of 2^8 .. 2^16, replayed from a graph
        dict(name="ensemble-48", kind="batch", runs=48, lo=256, hi=65536, grids=False, steps=16),
        # large single cells: 16 boxes of 2^20
        dict(name="boxes-1M", kind="batch", runs=16, lo=1048576, hi=1048576, grids=False, steps=2),
        # condensation on the grid with the condensed water of every cell
        dict(name="condense-256", kind="condense", nx=128, nz=128, per_cell=256, ragged=False),
        # the products of an output time
        dict(name="products-256", kind="products", nx=128, nz=128, per_cell=256, ragged=False),
        # a checkpoint of a sedimenting grid loaded again
        dict(name="restore-ragged", kind="restore", nx=64, nz=75, per_cell=203, ragged=True),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _grid_shape(rng, most):
    """A grid of at most `most` super-droplets, its cells of 24 to 420 on average."""
    per = _log_uniform(rng, 24, 420)
    nx = _log_uniform(rng, 8, 128)
    nz = max(4, min(160, _log_uniform(rng, 2000, most) // (per * nx)))
    return dict(nx=nx, nz=nz, per_cell=per, ragged=rng.random() < 0.7)


def draw(rng):
    kind = rng.choice(["cell", "box", "box", "grid", "grid", "coupled", "batch", "batch", "condense", "products",
                       "restore"])
    precision = rng.choice(["fp64", "fp64", "kfp32"])
    most = 128 * 128 * 256
    if kind == "cell":
        return dict(kind=kind, n_sd=2 * _log_uniform(rng, 32, 524288), precision=precision, dt=0.05,
                    kernel=rng.choice(["golovin", "geometric"]))
    if kind == "box":
        return dict(kind=kind, n_sd=_log_uniform(rng, 256, 1048576), steps=_log_uniform(rng, 4, 30),
                    host=rng.random() < 0.3, precision=precision)
    if kind == "grid":
        return dict(kind=kind, **_grid_shape(rng, most), developed=rng.random() < 0.6, steps=_log_uniform(rng, 2, 30),
                    one_call=rng.random() < 0.5, kernel=rng.choice(["geometric", "geometric", "long", "golovin"]),
                    precision=precision, cell_spectrum=rng.random() < 0.3)
    if kind == "coupled":
        return dict(kind=kind, **_grid_shape(rng, most), steps=rng.randint(2, 6), kernel=rng.choice(["geometric", "long"]),
                    precision=precision)
    if kind == "batch":
        if rng.random() < 0.3:  # a few large cells
            n = _log_uniform(rng, 20000, 1048576)
            return dict(kind=kind, runs=rng.randint(2, 8), lo=n // 2 + 1, hi=n, grids=False, steps=rng.randint(1, 4))
        return dict(kind=kind, runs=rng.randint(8, 56), lo=256, hi=_log_uniform(rng, 4096, 65536),
                    grids=rng.random() < 0.5, steps=rng.choice([4, 8, 16]))
    return dict(kind=kind, **_grid_shape(rng, most))


# ------------------------------------------------------------------ the inputs
def _device():
    return torch.device("cuda", torch.cuda.current_device())


def _gen(seed):
    g = torch.Generator(device=_device())
    g.manual_seed(int(seed) * 7919 + 17)
    return g


def _attributes(g, n, n_total, spectrum, developed):
    """xi (int64) and v (float64) of n super-droplets sampled at random, constant multiplicity but
    for a spread of a factor of three; developed: one in twelve is drizzle, few drops each."""
    u = torch.rand(n, generator=g, device=g.device, dtype=torch.float64)
    if spectrum == "exponential":
        v = -inputs.x0_box() * torch.log1p(-u * (1.0 - 1e-12)) + 1e-18
    else:
        z = torch.randn(n, generator=g, device=g.device, dtype=torch.float64).clamp_(-5.0, 5.0)
        r = inputs.LOGNORMAL_RADIUS * torch.exp(math.log(inputs.LOGNORMAL_SIGMA) * z)
        if developed:
            big = u < 1.0 / 12.0
            r = torch.where(big, 45.0e-6 * torch.exp(math.log(1.6) * z), r)
        v = (4.0 / 3.0 * math.pi) * r * r * r
    w = torch.rand(n, generator=g, device=g.device, dtype=torch.float64)
    mean = n_total / n
    xi = (mean * (0.5 + w)).round()
    if developed and spectrum != "exponential":
        xi = torch.where(u < 1.0 / 12.0, (xi * 1e-3).round(), xi)
    return xi.clamp_(min=1.0).to(torch.int64), v


def _cells(g, n_cells, per_cell, ragged):
    """Cell of every super-droplet, in increasing order: per_cell each, or sizes spread from a
    quarter of the mean to three times it (the same sizes for every seed, as the shape is the case's)."""
    if not ragged:
        return torch.arange(n_cells, device=g.device, dtype=torch.int32).repeat_interleave(per_cell)
    u = np.random.default_rng(n_cells + per_cell).random(n_cells)
    sizes = np.maximum(1, np.round(0.9 * per_cell * 0.25 * 12.0 ** u)).astype(np.int64)
    return torch.arange(n_cells, device=g.device, dtype=torch.int32).repeat_interleave(
        torch.as_tensor(sizes, device=g.device))


def _grid_inputs(case, seed, developed=True, spectrum="lognormal"):
    g = _gen(seed)
    n_cells = case["nx"] * case["nz"]
    cell = _cells(g, n_cells, case["per_cell"], case["ragged"])
    n = cell.numel()
    xi, v = _attributes(g, n, inputs.N_CONC_GRID * inputs.DV_GRID * n_cells, spectrum, developed)
    return g, n_cells, xi, v, cell


def _heights(g, cell, nx, dz):
    u = torch.rand(cell.numel(), generator=g, device=g.device, dtype=torch.float64)
    level = torch.div(cell, nx, rounding_mode="floor").to(torch.float64)
    return level * dz + u * (dz * 0.999)


def _fields(g, n_cells):
    """Growth coefficient and supersaturation of every cell (host arrays)."""
    u = torch.rand(n_cells, generator=g, device=g.device, dtype=torch.float64).cpu().numpy()
    return np.full(n_cells, 1.0e-10), 0.002 + 0.006 * u


def _batch_members(case):
    """(kernel, dt, dv, n_cells, n_sd, spectrum) of every run of a batch (sizes from the case alone)."""
    rng = np.random.default_rng(case["runs"] + case["hi"])
    out = []
    for i in range(case["runs"]):
        n = int(round(math.exp(rng.uniform(math.log(case["lo"]), math.log(case["hi"])))))
        dt = float(DT_CHOICES[int(rng.integers(3))])
        if case["grids"] and i % 2:
            cells = max(1, n // inputs.SD_PER_CELL_GRID)
            out.append(("geometric", dt, inputs.DV_GRID, cells, n, "lognormal"))
        else:
            out.append(("golovin", 0.25 * dt, inputs.DV_BOX, 1, n, "exponential"))
    return out


def _batch_inputs(case, seed):
    g = _gen(seed)
    for kernel, dt, dv, n_cells, n, spectrum in _batch_members(case):
        conc = inputs.N_CONC_BOX if kernel == "golovin" else inputs.N_CONC_GRID
        xi, v = _attributes(g, n, conc * dv * n_cells, spectrum, False)
        cell = (torch.arange(n, device=g.device, dtype=torch.int64) * n_cells // n).to(torch.int32)
        yield kernel, dt, dv, n_cells, xi, v, cell


def _box_inputs(case, seed):
    xi, v = _attributes(_gen(seed), case["n_sd"], inputs.N_CONC_BOX * inputs.DV_BOX, "exponential", False)
    return xi, v


def _cell_inputs(case, seed):
    if case["kernel"] == "golovin":
        return inputs.DV_BOX, *_attributes(_gen(seed), case["n_sd"], inputs.N_CONC_BOX * inputs.DV_BOX, "exponential",
                                           False)
    return inputs.DV_GRID, *_attributes(_gen(seed), case["n_sd"], inputs.N_CONC_GRID * inputs.DV_GRID, "lognormal", True)


def _restore_inputs(case, seed):
    g, n_cells, xi, v, cell = _grid_inputs(case, seed)
    z = _heights(g, cell, case["nx"], 10.0)
    order = torch.randperm(cell.numel(), generator=g, device=g.device)
    return n_cells, xi[order], v[order], cell[order].contiguous(), z[order]


def _new_run(kernel, precision, dt, dv, n_cells, seed, n):
    cfg = sdm.make_config(kernel, precision, dt=dt, dv=dv, n_cells=n_cells, seed=int(seed))
    return sdm.Run(cfg, n)


def _room(n):
    return (torch.empty(n, device=_device(), dtype=torch.int64), torch.empty(n, device=_device(), dtype=torch.float64))


def prepare(case, seed):
    kind = case["kind"]
    st = dict(case=case)
    if kind == "cell":
        dv, xi, v = _cell_inputs(case, seed)
        cfg = sdm.make_config(case["kernel"], case["precision"], dt=case["dt"], dv=dv, seed=int(seed))
        st.update(cfg=cfg, xi=xi, v=v, step=0, stream=sdm.current_stream_handle())
        return st
    if kind == "box":
        xi, v = _box_inputs(case, seed)
        n = case["n_sd"]
        cell = torch.zeros(n, device=xi.device, dtype=torch.int32)
        if case["host"]:
            xi, v, cell = xi.cpu().numpy(), v.cpu().numpy(), cell.cpu().numpy()
        else:
            st["out"] = _room(n)
        run = _new_run("golovin", case["precision"], 1.0, inputs.DV_BOX, 1, seed, n)
        st.update(run=run, xi=xi, v=v, cell=cell)
        return st
    if kind == "batch":
        runs = []
        total = sum(m[4] for m in _batch_members(case))
        st["out"] = _room(total)
        at, views = 0, []
        for i, (kernel, dt, dv, n_cells, xi, v, cell) in enumerate(_batch_inputs(case, seed)):
            n = xi.numel()
            run = _new_run(kernel, "fp64", dt, dv, n_cells, int(seed) * 1000 + i, n)
            runs.append(run.set_attributes(xi, v, cell))
            views.append((st["out"][0][at:at + n], st["out"][1][at:at + n]))
            at += n
        st.update(views=views, batch=sdm.Batch(runs, use_graph=True, graph_steps=case["steps"]))
        return st
    if kind == "restore":
        n_cells, xi, v, cell, z = _restore_inputs(case, seed)
        n = xi.numel()
        run = _new_run("geometric", "fp64", 1.0, inputs.DV_GRID, n_cells, seed, n)
        st.update(run=run, xi=xi, v=v, cell=cell, z=z, out=_room(n),
                  zc=(torch.empty(n, device=xi.device, dtype=torch.float64),
                      torch.empty(n, device=xi.device, dtype=torch.int32)))
        return st
    # the grids
    g, n_cells, xi, v, cell = _grid_inputs(case, seed, case.get("developed", True))
    n = xi.numel()
    run = _new_run(case.get("kernel", "geometric"), case.get("precision", "fp64"), 1.0, inputs.DV_GRID, n_cells, seed, n)
    st.update(run=run, xi=xi, v=v, cell=cell, n_cells=n_cells, out=_room(n))
    if kind == "grid" and case["cell_spectrum"] or kind == "products":
        st["spec"] = torch.empty(n_cells * (len(inputs.R_EDGES) - 1), device=xi.device, dtype=torch.float64)
    if kind == "coupled":
        st["z"] = _heights(g, cell, case["nx"], 10.0)
        st["zc"] = (torch.empty(n, device=xi.device, dtype=torch.float64),
                    torch.empty(n, device=xi.device, dtype=torch.int32))
    if kind in ("coupled", "condense"):
        st["G"], st["s"] = _fields(g, n_cells)
        st["water"] = [torch.empty(n_cells, device=xi.device, dtype=torch.float64) for _ in range(2)]
    if kind in ("condense", "products"):
        run.set_attributes(xi, v, cell)
    return st


# ------------------------------------------------------------------ one pass
def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "cell":
        sdm.sdm_cell_step_noalloc(st["cfg"], st["step"], st["xi"], st["v"], st["stream"])
        st["step"] += 1
        return {"xi": st["xi"], "v": st["v"]}
    if kind == "batch":
        st["batch"].step(case["steps"])
        for r, (xi, v) in zip(st["batch"].runs, st["views"]):
            sdm.sdm_get_attributes(r.h, xi=xi, volume=v)
        return {"xi": st["out"][0], "v": st["out"][1]}
    r = st["run"]
    if kind == "box":
        r.set_attributes(st["xi"], st["v"], st["cell"])
        r.step(case["steps"])
        spec = r.spectrum(inputs.R_EDGES)
        if case["host"]:
            xi, v = r.attributes()
        else:
            xi, v = sdm.sdm_get_attributes(r.h, xi=st["out"][0], volume=st["out"][1])
        return {"spectrum": spec, "xi": xi, "v": v}
    if kind == "grid":
        r.set_attributes(st["xi"], st["v"], st["cell"])
        if case["one_call"]:
            r.step(case["steps"])
        else:
            for _ in range(case["steps"]):
                r.step(1)
        if case["cell_spectrum"]:
            spec = r.spectrum(inputs.R_EDGES, per_cell=True, out=st["spec"])
        else:
            spec = r.spectrum(inputs.R_EDGES)
        xi, v = sdm.sdm_get_attributes(r.h, xi=st["out"][0], volume=st["out"][1])
        return {"spectrum": spec, "xi": xi, "v": v}
    if kind == "coupled":
        r.set_attributes(st["xi"], st["v"], st["cell"])
        r.set_positions(st["z"], nx=case["nx"], dz=10.0)
        fallen = 0.0
        for _ in range(case["steps"]):
            r.step(1)
            sdm.sdm_condensation_step(r.h, st["G"], st["s"], R_MIN, n_cells=st["n_cells"], out=st["water"][0])
            fallen += r.sediment()
        xi, v = sdm.sdm_get_attributes(r.h, xi=st["out"][0], volume=st["out"][1])
        z, cell = sdm.sdm_get_positions(r.h, z=st["zc"][0], cell=st["zc"][1])
        return {"fallen": fallen, "xi": xi, "v": v, "z": z, "cell": cell, "water": st["water"][0]}
    if kind == "condense":
        up = sdm.sdm_condensation_step(r.h, st["G"], st["s"], R_MIN, n_cells=st["n_cells"], out=st["water"][0])
        down = sdm.sdm_condensation_step(r.h, st["G"], -st["s"], R_MIN, n_cells=st["n_cells"], out=st["water"][1])
        _, v = sdm.sdm_get_attributes(r.h, volume=st["out"][1])
        return {"up": up, "down": down, "v": v}
    if kind == "products":
        total = r.spectrum(inputs.R_EDGES)
        cells = r.spectrum(inputs.R_EDGES, per_cell=True, out=st["spec"])
        d = r.diagnostics()
        return {"total": total, "cells": cells, "live": d["live_sd"], "xi": d["sum_xi"], "water": d["sum_xi_v"]}
    if kind == "restore":
        r.set_attributes(st["xi"], st["v"], st["cell"])
        r.set_positions(st["z"], nx=case["nx"], dz=10.0)
        z, cell = sdm.sdm_get_positions(r.h, z=st["zc"][0], cell=st["zc"][1])
        xi, v = sdm.sdm_get_attributes(r.h, xi=st["out"][0], volume=st["out"][1])
        return {"xi": xi, "v": v, "z": z, "cell": cell}
    raise ValueError(kind)


# ------------------------------------------------------------------ what it cannot do without
def work(case):
    """Bytes: inputs read once and outputs written once (xi and v are 16 B per super-droplet, the
    cell 4, a height 8).  Flops: per super-droplet and step three quarters of a Philox block
    (about 100 integer operations), some 40 for ordering and 30 for its half of a pair."""
    kind = case["kind"]
    per_step = 145.0
    nb = len(inputs.R_EDGES) - 1
    if kind == "cell":
        return {"bytes": 16.0 * case["n_sd"], "flops": per_step * case["n_sd"]}
    if kind == "box":
        n = case["n_sd"]
        return {"bytes": 36.0 * n + 8.0 * nb, "flops": per_step * n * case["steps"]}
    if kind == "batch":
        n = sum(m[4] for m in _batch_members(case))
        return {"bytes": 32.0 * n, "flops": per_step * n * case["steps"]}
    n_cells = case["nx"] * case["nz"]
    n = n_cells * case["per_cell"]
    if kind == "grid":
        spec = 8.0 * nb * (n_cells if case["cell_spectrum"] else 1)
        steps = case["steps"]
        own = 0.0 if case["one_call"] else 16.0 * n * steps
        return {"bytes": 36.0 * n + spec + own, "flops": per_step * n * steps}
    if kind == "coupled":
        # attributes and heights in and out; per step the state read for coalescence, read and v
        # written for condensation, and the layout (32 B) read and written for sedimentation
        return {"bytes": n * (28.0 + 28.0 + case["steps"] * (16.0 + 24.0 + 64.0)),
                "flops": n * case["steps"] * (per_step + 60.0 + 40.0)}
    if kind == "condense":
        return {"bytes": 2 * 24.0 * n + 16.0 * n + 32.0 * n_cells, "flops": 2 * 60.0 * n}
    if kind == "products":
        return {"bytes": 3 * 16.0 * n + 8.0 * nb * (n_cells + 1), "flops": 2 * 40.0 * n + 4.0 * n}
    return {"bytes": 56.0 * n, "flops": 2.0 * n}


# ------------------------------------------------------------------ the same in 64 bits
_M32 = 0xFFFFFFFF


def _philox(c0, c1, c2, c3, k0, k1):
    """Philox4x32-10 on int64 tensors or numbers holding 32-bit words."""
    c0, c1 = torch.broadcast_tensors(c0, c1)
    c2 = torch.full_like(c0, c2)
    c3 = torch.full_like(c0, c3)
    for r in range(10):
        p0, p1 = c0 * 0xD2511F53, c2 * 0xCD9E8D57
        c0, c1, c2, c3 = (((p1 >> 32) & _M32) ^ c1 ^ k0, p1 & _M32, ((p0 >> 32) & _M32) ^ c3 ^ k1, p0 & _M32)
        k0, k1 = (k0 + 0x9E3779B9) & _M32, (k1 + 0xBB67AE85) & _M32
    return c0, c1, c2, c3


def _words(index, cell, step, tag, seed):
    """The 64-bit draw of every (index, cell), as two 32-bit words."""
    w = _philox(index >> 1, cell, step & _M32, ((step >> 32) & 0x7FFFFFFF) | (tag << 31), seed & _M32,
                (seed >> 32) & _M32)
    odd = (index & 1).bool()
    return torch.where(odd, w[2], w[0]), torch.where(odd, w[3], w[1])


def _speed(r):
    return torch.where(r < 40.0e-6, 1.19e8 * r * r, torch.where(r < 600.0e-6, 8.0e3 * r, 201.0 * torch.sqrt(r)))


def _kernel(kernel, vj, vk):
    if kernel == "golovin":
        return inputs.GOLOVIN_B * (vj + vk)
    rj, rk = (0.75 / math.pi * vj) ** (1.0 / 3.0), (0.75 / math.pi * vk) ** (1.0 / 3.0)
    k = math.pi * (rj + rk) ** 2 * (_speed(rj) - _speed(rk)).abs()
    if kernel == "long":
        big, small = torch.maximum(rj, rk), torch.minimum(rj, rk)
        e = (4.5e8 * big * big * (1.0 - 3e-6 / small)).clamp(min=1e-3)
        k = k * torch.where(big > 50e-6, torch.ones_like(e), e)
    return k


def _coalesce(xi, v, cell, n_cells, kernel, dt, dv, seed, first, steps):
    """`steps` coalescence steps of super-droplets in cell order (in place)."""
    total = torch.bincount(cell.long(), minlength=n_cells)
    start = torch.cumsum(total, 0) - total
    rank = torch.arange(xi.numel(), device=xi.device) - start[cell.long()]
    for s in range(first, first + steps):
        live = (xi > 0).nonzero().squeeze(1)
        c = cell[live].long()
        hi, lo = _words(rank[live], c, s, 0, seed)
        order = torch.sort((hi << 32 | lo) ^ (-1 << 63), stable=True).indices
        order = order[torch.sort(c[order], stable=True).indices]
        who = live[order]
        n_c = torch.bincount(c, minlength=n_cells)
        at = torch.cumsum(n_c, 0) - n_c
        pairs = n_c // 2
        pc = torch.repeat_interleave(torch.arange(n_cells, device=xi.device), pairs)
        l = torch.arange(pc.numel(), device=xi.device) - (torch.cumsum(pairs, 0) - pairs)[pc]
        a, b = who[at[pc] + 2 * l], who[at[pc] + 2 * l + 1]
        swap = xi[a] < xi[b]
        j, k = torch.where(swap, b, a), torch.where(swap, a, b)
        n = n_c[pc].double()
        p = _kernel(kernel, v[j], v[k]) * xi[j].double() * (dt / dv * (n * (n - 1.0) / 2.0 / pairs[pc].double()))
        wa, wb = _words(l, pc, s, 1, seed)
        u = ((wa << 21) | (wb >> 11)).double() * 2.0 ** -53
        g = torch.ceil(p - u)
        cap = torch.div(xi[j], xi[k], rounding_mode="floor")
        hit = g >= 1.0
        j, k, g, cap = j[hit], k[hit], g[hit], cap[hit]
        g = torch.where(g >= cap.double(), cap, g.clamp(max=9e18).long())
        vn = v[k] + g.double() * v[j]
        left = xi[j] - g * xi[k]
        split = left == 0
        half = torch.div(xi[k], 2, rounding_mode="floor")
        xk = xi[k]
        xi[j] = torch.where(split, half, left)
        xi[k] = torch.where(split, xk - half, xk)
        v[j] = torch.where(split, vn, v[j])
        v[k] = vn
    return xi, v


def _spectrum(xi, v, cell, n_cells, dv, per_cell):
    e = torch.as_tensor(inputs.R_EDGES, device=xi.device, dtype=torch.float64)
    nb = e.numel() - 1
    r = (0.75 / math.pi * v) ** (1.0 / 3.0)
    b = torch.searchsorted(e, r, right=True) - 1
    ok = (b >= 0) & (b < nb) & (xi > 0)
    w = (xi.double() * v)[ok]
    dln = torch.log(e[1:]) - torch.log(e[:-1])
    if per_cell:
        acc = torch.bincount(cell[ok].long() * nb + b[ok], weights=w, minlength=n_cells * nb)
        return (acc.view(n_cells, nb) / dv / dln).reshape(-1)
    return torch.bincount(b[ok], weights=w, minlength=nb) / (dv * n_cells) / dln


def _grow(v, cell, G, s, dt):
    r2 = ((0.75 / math.pi * v) ** (1.0 / 3.0)) ** 2
    c = torch.as_tensor(2.0 * G * s * dt, device=v.device)[cell.long()]
    new = torch.maximum(r2 + c, r2.clamp(max=R_MIN * R_MIN))
    dvol = 4.0 / 3.0 * math.pi * (new - r2) * (new + torch.sqrt(new * r2) + r2) / (torch.sqrt(new) + torch.sqrt(r2))
    return v + dvol, dvol


def exact(case, seed):
    kind = case["kind"]
    if case.get("precision") == "kfp32" or kind == "coupled":
        return None  # the step itself is defined in binary32 there
    if kind == "cell":
        dv, xi, v = _cell_inputs(case, seed)
        xi, v = _coalesce(xi, v, torch.zeros_like(xi), 1, case["kernel"], case["dt"], dv, int(seed), 0, 1)
        return {"xi": xi, "v": v}
    if kind == "box":
        xi, v = _box_inputs(case, seed)
        cell = torch.zeros_like(xi)
        xi, v = _coalesce(xi, v, cell, 1, "golovin", 1.0, inputs.DV_BOX, int(seed), 0, case["steps"])
        return {"spectrum": _spectrum(xi, v, cell, 1, inputs.DV_BOX, False), "xi": xi, "v": v}
    if kind == "batch":
        done = [_coalesce(xi, v, cell, n_cells, kernel, dt, dv, int(seed) * 1000 + i, 0, case["steps"])
                for i, (kernel, dt, dv, n_cells, xi, v, cell) in enumerate(_batch_inputs(case, seed))]
        return {"xi": torch.cat([d[0] for d in done]), "v": torch.cat([d[1] for d in done])}
    if kind == "restore":
        n_cells, xi, v, cell, z = _restore_inputs(case, seed)
        return {"xi": xi, "v": v, "z": z, "cell": cell}
    g, n_cells, xi, v, cell = _grid_inputs(case, seed, case.get("developed", True))
    dv = inputs.DV_GRID
    if kind == "grid":
        xi, v = _coalesce(xi, v, cell, n_cells, case["kernel"], 1.0, dv, int(seed), 0, case["steps"])
        return {"spectrum": _spectrum(xi, v, cell, n_cells, dv, case["cell_spectrum"]), "xi": xi, "v": v}
    if kind == "condense":
        G, s = _fields(g, n_cells)
        water = []
        for sign in (1.0, -1.0):
            v, dvol = _grow(v, cell, G, sign * s, 1.0)
            water.append(torch.bincount(cell.long(), weights=xi.double() * dvol, minlength=n_cells))
        return {"up": water[0], "down": water[1], "v": v}
    return {"total": _spectrum(xi, v, cell, n_cells, dv, False), "cells": _spectrum(xi, v, cell, n_cells, dv, True),
            "live": int((xi > 0).sum()), "xi": int(xi.sum()), "water": float((xi.double() * v).sum())}
