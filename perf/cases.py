"""The calls whose time matters: what users of this package have it do, through
its public entry points (``System``, ``Batch``), from the smallest melt to the
134M-particle one.

Each case is one system (or batch) and one pass over it: a number of SCMF
cycles followed by a read of the new configuration, a training call of the
learned proposal, or the analysis of a given configuration.  The sizes are the
ones of ``paper_1711_03828_gb300.workloads``, the paper's printed thin film,
and boxes of the same density between them.

A Metropolis trajectory has no 64-bit value to compare with after several
cycles (a decision within rounding of its threshold changes the fields, and
with them every later decision), so ``exact`` covers the analysis cases.
"""
from __future__ import annotations

import dataclasses
import math

import numpy as np
import torch

from paper_1711_03828_gb300 import (Batch, GRID_BF16, GRID_F16, GRID_F32, ITERATION_MOLECULE,
                                    MOVE_LEARNED, MOVE_SMC, MOVE_UNIFORM, SET_ORDER_RANDOM, System,
                                    SystemDesc, workloads)

MOVES = {"uniform": MOVE_UNIFORM, "smc": MOVE_SMC, "learned": MOVE_LEARNED}
GRIDS = {"f32": GRID_F32, "bf16": GRID_BF16, "f16": GRID_F16}
L2_BYTES = 129e6    # a configuration larger than this streams from memory every cycle


def _case(kind, N, grid, cycles, *, name=None, per_Re=6, rho=4096.0, f=0.5, chiN=30.0, move="uniform",
          iteration="set", dtype="f32", **more):
    c = dict(kind=kind, N=N, gx=grid[0], gy=grid[1], gz=grid[2], cycles=cycles, per_Re=per_Re, rho=rho,
             f=f, chiN=chiN, move=move, iteration=iteration, dtype=dtype, **more)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the first thing anyone runs: 32,768 particles, 100 cycles (latency and launches)
        _case("melt", 32, (12, 12, 12), 100, chiN=20.0, name="melt_small"),
        # the production melt: 134,217,728 particles
        _case("melt", 32, (192, 192, 192), 16, name="melt_large"),
        # the slow melt (chains of 64) with force-biased moves, 67,108,864 particles
        _case("melt", 64, (192, 192, 96), 16, chiN=40.0, move="smc", name="melt_slow_smc"),
        # its 8x8x4 R_e0 box under the learned proposal: ten cycles between two samples
        _case("melt", 64, (48, 48, 24), 10, chiN=40.0, move="learned", name="learned_box"),
        # the paper's lamellar thin film (N = 100, 1.2 R_e0 thick, walls that attract A), a
        # 40 x 40 R_e0 piece with ten cells per R_e0, 16-bit fields
        _case("film", 100, (400, 400, 12), 16, per_Re=10, rho=8570.0, dtype="bf16", name="thin_film"),
        # chains of odd length under force-biased moves, 16-bit fields
        _case("melt", 33, (48, 48, 48), 20, move="smc", dtype="f16", name="odd_smc"),
        # the molecule-parallel iteration at an ordinary size
        _case("melt", 32, (48, 48, 48), 20, iteration="molecule", name="molecule_parallel"),
        # stars, combs, rings and diblocks mixed, 16,777,216 particles
        _case("arch", 32, (96, 96, 96), 16, name="arch_mid"),
        # three particle types, triblocks, stars and rings, force-biased moves
        _case("abc", 32, (48, 48, 48), 20, move="smc", name="abc_smc"),
        # 64 systems of uneven size advanced together
        _case("batch", 0, (0, 0, 0), 64, members=64, layout=1, name="batch64"),
        # what is read off a configuration: fields, energies, R_e^2, S(q) at 64 wave vectors
        _case("analysis", 32, (96, 96, 96), 0, waves=64, name="analysis"),
        # training the learned proposal on plain trajectories of the 8x8x4 box
        _case("train", 64, (48, 48, 24), 5, chiN=40.0, move="learned", steps=8, samples=16384,
              name="train"),
    ]


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _box(rng, particles, rho=4096.0, per_Re=6, layers=None):
    """Grid of about the given number of particles, every edge its own length."""
    cells = particles / rho * per_Re ** 3
    if layers:
        edge = math.sqrt(cells / layers)
        s = rng.uniform(0.7, 1.4)
        return max(2, round(edge * s)), max(2, round(edge / s)), layers
    edge = cells ** (1.0 / 3.0)
    a, b = rng.uniform(0.75, 1.3), rng.uniform(0.75, 1.3)
    return max(2, round(edge * a)), max(2, round(edge * b)), max(2, round(edge / (a * b)))


def draw(rng):
    chiN = rng.uniform(10.0, 40.0)
    f = rng.choice([0.3, 0.5, 0.7])
    dtype = rng.choice(["f32", "f32", "bf16", "f16"])
    # single cycles, samples of ten, graph-sized runs and runs with a remainder
    cycles = rng.choice([1, 5, 10, 16, 20, 37])
    kind = rng.choice(["melt", "melt", "melt", "smc", "smc", "learned", "film", "molecule", "arch",
                       "abc", "batch", "analysis", "train"])
    even = rng.choice([8, 16, 32, 64])
    if kind == "melt":
        N = rng.choice([even, even, 2 * rng.randint(1, 31) + 1])
        return _case("melt", N, _box(rng, _log_uniform(rng, 4096, 6e7)), cycles, f=f, chiN=chiN,
                     dtype=dtype)
    if kind == "smc":
        N = rng.choice([even, 2 * rng.randint(1, 31) + 1, rng.randint(65, 130)])
        return _case("melt", N, _box(rng, _log_uniform(rng, 4096, 2e7)), cycles, f=f, chiN=chiN,
                     move="smc", dtype=dtype)
    if kind == "learned":
        return _case("melt", even, _box(rng, _log_uniform(rng, 3e4, 4e6)), cycles, f=f, chiN=chiN,
                     move="learned", dtype=dtype)
    if kind == "film":
        return _case("film", rng.randint(65, 200),
                     _box(rng, _log_uniform(rng, 1e5, 1.6e7), 8570.0, 10, rng.randint(8, 14)), cycles,
                     per_Re=10, rho=8570.0, f=f, chiN=chiN, dtype=dtype)
    if kind == "molecule":
        return _case("melt", rng.randint(8, 64), _box(rng, _log_uniform(rng, 8192, 4e6)), cycles, f=f,
                     chiN=chiN, iteration="molecule", dtype=dtype)
    if kind in ("arch", "abc"):
        return _case(kind, 32, _box(rng, _log_uniform(rng, 3e4, 1.6e7)), cycles, chiN=chiN,
                     move=rng.choice(["uniform", "smc"]), dtype="f32" if kind == "abc" else dtype)
    if kind == "batch":
        return _case("batch", 0, (0, 0, 0), 16 * rng.randint(1, 4), members=rng.randint(8, 64),
                     layout=rng.randint(2, 999), dtype=dtype)
    if kind == "analysis":
        return _case("analysis", rng.randint(8, 100), _box(rng, _log_uniform(rng, 3e4, 1.6e7)), 0, f=f,
                     chiN=chiN, waves=rng.randint(1, 100))
    return _case("train", even, _box(rng, _log_uniform(rng, 3e4, 2e6)), rng.randint(1, 5), f=f,
                 chiN=chiN, move="learned", steps=rng.randint(2, 8), samples=rng.randint(1000, 16384))


def _grid(case):
    return case["gx"], case["gy"], case["gz"]


def _cells(case):
    return case["gx"] * case["gy"] * case["gz"]


def _chains(case):
    return max(1, round(case["rho"] * _cells(case) / case["per_Re"] ** 3 / case["N"]))


def _desc(case, seed):
    return SystemDesc(n_chains=_chains(case), N=case["N"], f=case["f"],
                      box_Re=tuple(g / case["per_Re"] for g in _grid(case)), grid=_grid(case),
                      chiN=case["chiN"], kappaN=50.0, move=MOVES[case["move"]],
                      set_order=ITERATION_MOLECULE if case["iteration"] == "molecule" else SET_ORDER_RANDOM,
                      grid_dtype=GRIDS[case["dtype"]], seed=seed % (1 << 62))


def _members(case, seed):
    return [dataclasses.replace(d, seed=seed % (1 << 62))
            for d in workloads.batch_replicas(case["members"], seed=case["layout"],
                                              grid_dtype=GRIDS[case["dtype"]])]


def _walks(parent, n, case, g):
    """Gaussian molecules on the GPU: particle i at its parent plus a bond, one without a parent
    anywhere in the box; (3, n, N) float32."""
    N = len(parent)
    sigma = case["per_Re"] / math.sqrt(3.0 * max(N - 1, 1))
    box = torch.tensor(_grid(case), dtype=torch.float32, device="cuda").reshape(3, 1)
    out = torch.empty((3, n, N), dtype=torch.float32, device="cuda")
    for i, p in enumerate(parent):
        if p < 0:
            out[:, :, i] = torch.rand((3, n), generator=g, device="cuda") * box
        else:
            out[:, :, i] = out[:, :, p] + sigma * torch.randn((3, n), generator=g, device="cuda")
    return out


def _parents(molecule, N):
    parent = [-1] * N
    for i, j in molecule[1]:
        a, b = min(i, j), max(i, j)
        if parent[b] < 0 or a < parent[b]:
            parent[b] = a
    return parent


def _linear(case, seed):
    """Chains of an analysis case, in the spatial order a relabelled configuration has."""
    g = torch.Generator(device="cuda").manual_seed(seed % (1 << 62))
    pos = _walks([-1] + list(range(case["N"] - 1)), _chains(case), case, g)
    block = (pos[:, :, 0] / 8.0).long()
    order = torch.argsort((block[2] * 4096 + block[1]) * 4096 + block[0], stable=True)
    return pos[:, order].reshape(3, -1).contiguous()


def _waves(case, seed):
    """Low wave vectors, as a search for the strongest mode asks for them."""
    r = np.random.default_rng(seed)
    m = r.integers(-6, 7, size=(case["waves"], 3)).astype(np.int32)
    m[(m == 0).all(axis=1)] = (1, 0, 0)
    return m


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        batch = Batch(_members(case, seed))
        pos = torch.empty(3 * batch.M, dtype=torch.float32, device="cuda")
        dens = torch.empty(sum(d.cells for d in batch.descs), dtype=torch.int32, device="cuda")
        views, a, b = [], 0, 0
        for m in batch.members:
            views.append((m, pos[a:a + 3 * m.desc.M], dens[b:b + m.desc.cells]))
            a, b = a + 3 * m.desc.M, b + m.desc.cells
        return dict(case=case, batch=batch, views=views, pos=pos, dens=dens)
    d = _desc(case, seed)
    state = dict(case=case)
    if kind == "analysis":
        state.update(given=_linear(case, seed), waves=_waves(case, seed))
        d.flags = 1    # SOMA_FLAG_NO_SORT: the configuration is given
    s = System(d)
    if kind == "film":
        # walls: nothing enters the outer layers, and A is attracted to the next ones
        z = torch.arange(d.grid[2], device="cuda").repeat_interleave(d.grid[0] * d.grid[1])
        wall = (z == 0) | (z == d.grid[2] - 1)
        near = (z == 1) | (z == d.grid[2] - 2)
        ext = torch.stack([near * -0.1, near * 0.0]).to(torch.float32).contiguous()
        forbidden = wall.to(torch.uint8).contiguous()
        torch.cuda.synchronize()
        s.set_external(ext, forbidden)
        s.update_fields()
    elif kind in ("arch", "abc"):
        if kind == "abc":
            mols = workloads.abc_molecules()
            s.set_types(3, workloads.ABC_CHI_N)
        else:
            mols = workloads.arch_large_molecules()
        words, starts = workloads.encode_architectures(mols)
        g = torch.Generator(device="cuda").manual_seed(seed % (1 << 62))
        arch = torch.randint(len(mols), (d.n_chains,), generator=g, device="cuda")
        pos = torch.empty((3, d.n_chains, d.N), dtype=torch.float32, device="cuda")
        for k, mol in enumerate(mols):
            at = (arch == k).nonzero()[:, 0]
            pos[:, at] = _walks(_parents(mol, d.N), at.numel(), case, g)
        s.set_topology(words, starts, arch.to(torch.uint8).cpu().numpy())
        torch.cuda.synchronize()
        s.set_positions(pos.reshape(3, -1))
        s.sort_molecules()
        s.update_fields()
    if case["move"] == "learned":
        s.set_proposal_weights(workloads.random_mlp(seed % (1 << 31)))
    state["system"] = s
    if kind != "analysis":
        state["pos"] = torch.empty(3 * d.M, dtype=torch.float32, device="cuda")
    if kind != "abc":
        state["dens"] = torch.empty(d.cells, dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()
    return state


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "batch":
        state["batch"].sweep(case["cycles"])
        for m, pos, dens in state["views"]:
            m.get_positions(out=pos)
            m.get_density(out=dens)
        return {"positions": state["pos"], "density": state["dens"]}
    s = state["system"]
    if kind == "analysis":
        s.set_positions(state["given"])
        s.update_fields()
        return {"observables": s.observables(), "sq": s.structure_factor(state["waves"]),
                "density": s.get_density(out=state["dens"])}
    if kind == "train":
        log = s.train_proposal(steps=case["steps"], batch=case["samples"], sweeps_between=case["cycles"],
                               lr=3e-3)
        return {"weights": s.get_proposal_weights(), "log": log,
                "positions": s.get_positions(out=state["pos"]),
                "density": s.get_density(out=state["dens"])}
    s.sweep(case["cycles"])
    pos = s.get_positions(out=state["pos"])
    if kind == "abc":
        return {"positions": pos, "counts": s.get_type_counts()}
    return {"positions": pos, "density": s.get_density(out=state["dens"])}


def work(case):
    """Each position in and out once per cycle where the configuration exceeds
    the L2 cache, else once per pass; each grid likewise (occupation numbers
    out, fields in).  Operations: the energy change, trial position and cell of
    a move, the field force of a force-biased one, the network (and its
    gradient) of a learned one."""
    if case["kind"] == "batch":
        descs = _members(case, 1)
        M, cells, cycles = sum(d.M for d in descs), sum(d.cells for d in descs), case["cycles"]
    else:
        M, cells, cycles = _chains(case) * case["N"], _cells(case), case["cycles"]
    field = 4 if case["dtype"] == "f32" else 2
    types = 3 if case["kind"] == "abc" else 2
    if case["kind"] == "analysis":
        # positions and wave vectors in, counts out; bond and end-to-end sums, S(q) by cells
        return {"bytes": 12.0 * M + 4.0 * cells, "flops": 11.0 * M + 2.0 * cells * case["waves"]}
    grids = cells * (types * field + 4.0)
    once = 24.0 * M + grids
    passes = case["steps"] * cycles if case["kind"] == "train" else cycles
    net = 2 * (12 * 32 + 32 * 32 + 32 * 4)
    per_move = {"uniform": 40.0, "smc": 110.0, "learned": 110.0 + 2 * net}[case["move"]]
    if case["kind"] == "train":
        flops = passes * M * 40.0 + case["steps"] * case["samples"] * 6.0 * net
    else:
        flops = passes * M * per_move
    return {"bytes": once * (passes if once > L2_BYTES else 1), "flops": flops}


def exact(case, seed):
    """The analysis of the given configuration in 64 bits: counts by floor and
    modulo, the energies and R_e^2 of their definitions, S(q) by the FFT."""
    if case["kind"] != "analysis":
        return None
    N, n = case["N"], _chains(case)
    gx, gy, gz = _grid(case)
    r = _linear(case, seed).double().reshape(3, n, N)
    c = torch.floor(r).long()
    cell = ((c[2] % gz) * gy + c[1] % gy) * gx + c[0] % gx
    n_a = math.floor(case["f"] * N + 0.5)
    counts = [torch.bincount(part.reshape(-1), minlength=gx * gy * gz).double()
              for part in (cell[:, :n_a], cell[:, n_a:])]
    rho_cell = n * N / (gx * gy * gz)
    phi = [k / rho_cell for k in counts]
    K = 25.0 * (phi[0] + phi[1] - 1.0) ** 2 - 0.25 * case["chiN"] * (phi[0] - phi[1]) ** 2
    E_nb = rho_cell / N * float(K.sum())
    Re = float(case["per_Re"])
    b2 = float((r[:, :, 1:] - r[:, :, :-1]).square().sum())
    E_b = 3.0 * (N - 1) / (2.0 * Re * Re) * b2
    Re2 = float((r[:, :, -1] - r[:, :, 0]).square().sum()) / n
    m = torch.as_tensor(_waves(case, seed), device="cuda").long()
    F = torch.fft.fftn((counts[0] - counts[1]).reshape(gz, gy, gx))
    sq = F[m[:, 2] % gz, m[:, 1] % gy, m[:, 0] % gx].abs().square() / (n * N)
    return {"observables": {"E_b": E_b, "E_nb": E_nb, "E_tot": E_b + E_nb, "Re2": Re2,
                            "Re2_rel": Re2 / (Re * Re), "b2": b2 / max(n * (N - 1), 1),
                            "accepted": None, "attempted": None, "sweeps": None, "max_cell": None,
                            "E_ext": 0.0},
            "sq": sq, "density": None}
