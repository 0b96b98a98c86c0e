"""The performance cases of this framework: the work its users have it do.

A case is a dict of plain values.  ``prepare`` makes what a user's program
holds before the timed call (tissues with their state on the GPU, a batch, a
server's requests), ``run`` is one pass through the public entry points, and
``work`` the bytes and operations that pass cannot do without.

Kinds:
  tissue   one tissue advanced by Tissue.step, the state left on the device;
           with io = 1 the state comes from pinned host memory and goes back
           to it around the step, with stats = 1 the program also reads the
           per-cell event counts and times, as one that watches a run does
  batch    many tissues advanced by one Batch.step
  serving  a whole Server.run over requests that are waiting at its start

States: Notch-Delta tissues mid-run hold tens of molecules per voxel (about
60 D, 30 N and 10 R after 20 time units with the default rates; a batch that
is 5 time units old has about 4 kD + 3 D, 22 N and 4 R), promoter tissues
about 0.2 Delta and 0.05 NICD.  Counts are drawn from Poisson laws of those
means, so a pass meets the event rates of a running simulation.
"""
from __future__ import annotations

import math
from dataclasses import replace

import numpy as np
import torch

from paper_1806_10889_gb300 import workloads as W
from paper_1806_10889_gb300.batching import Batch
from paper_1806_10889_gb300.serving import Server
from paper_1806_10889_gb300.tissue import SPLIT_STRANG, Tissue

RUNNING = (60.0, 30.0, 10.0)  # D, N, R per voxel of a Notch-Delta tissue mid-run
YOUNG = (22.0, 13.0, 4.0)     # after 2 time units
START = (5.0, 5.0, 5.0)       # its initial state
EVENTS_MAX = 6.0e8            # most chi events of a drawn case's pass


def _tissue(name, width, height, n, dt, steps=1, model="nd", state="running", strang=0, k_in=0.0,
            k_off=0.0, edge=-1, io=0, stats=0):
    return dict(name=name, kind="tissue", width=width, height=height, n=n, dt=dt, steps=steps,
                model=model, state=state, strang=strang, k_in=k_in, k_off=k_off, edge=edge, io=io,
                stats=stats)


def listed():
    return [
        # the smallest configuration of the suite: an interactive run that
        # looks at every step
        _tissue("tiny", 2, 2, 8, 0.1, stats=1),
        # a short step on few cells: launches and the host path count
        _tissue("short_step", 6, 4, 16, 0.001, steps=4),
        # ragged cells (not a multiple of 4 voxels), binding inside the voxel,
        # Strang splitting: a convergence study
        _tissue("ragged_strang", 23, 17, 21, 0.05, strang=1, k_in=0.001, k_off=0.5),
        # the medium configuration at the suite's two shorter step lengths,
        # the longer one end to end through pinned host memory
        _tissue("medium", 64, 64, 16, 0.1, io=1),
        _tissue("medium_fine_steps", 64, 64, 16, 0.01, steps=5),
        # the paper's own model, and with well-mixed interior cells
        _tissue("promoter", 64, 64, 16, 0.1, model="promoter"),
        _tissue("mixed_fidelity", 64, 64, 16, 0.1, model="promoter", edge=8),
        # a wide layer of small cells
        _tissue("wide_small_cells", 256, 256, 8, 0.1),
        # an ordinary tissue of the largest cells
        _tissue("big_cells", 48, 48, 32, 0.1, stats=1),
        # the large configuration: 256x256 cells of 32x32 voxels, 2 time units old
        _tissue("large", 256, 256, 32, 0.1, state="young"),
        # uneven tissues of three cell sizes advanced together (a parameter
        # sweep), from the generator of the 256-tissue configuration
        dict(name="uneven_batch", kind="batch", members=60, dt=0.1, steps=1, strang=0),
        # a service's first chunk: requests of several replicas, results read back
        dict(name="serving", kind="serving", first=0, requests=10, replicas=4, steps=5, dt=0.1),
    ]


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["tissue", "tissue", "tissue", "tissue", "batch", "serving"])
    if kind == "batch":
        return dict(kind="batch", members=rng.randint(3, 60), dt=_log_uniform(rng, 0.01, 0.1),
                    steps=rng.randint(1, 3), strang=rng.randint(0, 1))
    if kind == "serving":
        return dict(kind="serving", first=rng.randint(0, 480), requests=rng.randint(1, 12),
                    replicas=rng.randint(1, 6), steps=rng.randint(1, 8),
                    dt=_log_uniform(rng, 0.02, 0.1))
    while True:
        model = rng.choice(["nd", "nd", "nd", "nd", "promoter"])
        binding = model == "nd" and rng.random() < 0.2
        c = _tissue("", max(1, round(_log_uniform(rng, 1.0, 256.9))),
                    max(1, round(_log_uniform(rng, 1.0, 256.9))),
                    rng.choice([8, 16, 32, rng.randint(2, 32)]), _log_uniform(rng, 0.001, 1.0),
                    steps=rng.randint(1, 4), model=model,
                    state=rng.choice(["start", "young", "running", "running"]),
                    strang=int(rng.random() < 0.25), k_in=0.001 if binding else 0.0,
                    k_off=0.5 if binding else 0.0,
                    edge=rng.randint(1, 8) if model == "promoter" and rng.random() < 0.4 else -1,
                    io=int(rng.random() < 0.2), stats=int(rng.random() < 0.3))
        del c["name"]
        # no more than the largest listed case, and no cell alone with a chain
        # of events longer than a second
        if _events(c) <= EVENTS_MAX and _events(c) / (c["width"] * c["height"]) <= 3.0e5:
            return c


def _spec(c, seed):
    model = W.promoter_model(c["n"]) if c["model"] == "promoter" else dict(
        W.ND_MODEL, k_in=c["k_in"], k_off=c["k_off"])
    return W.TissueSpec(c["width"], c["height"], c["n"], seed=1 + seed, tissue_id=0, model=model,
                        init_lambda=(0.2, 0.05, 0.0) if c["model"] == "promoter" else START,
                        fidelity="lattice" if c["edge"] < 0 else f"edge:{c['edge']}")


def _means(c):
    if c["model"] == "promoter":
        return (0.2, 0.05, 0.0)
    return {"running": RUNNING, "young": YOUNG, "start": START}[c["state"]]


def _fill(buffer, cells, V, means, gen):
    """Poisson counts of the given means into a state buffer, a few million at a time."""
    view = buffer.view(cells, 3, V)
    lam = torch.tensor(means, device="cuda", dtype=torch.float32).view(1, 3, 1)
    chunk = max(1, (1 << 24) // (3 * V))
    for i in range(0, cells, chunk):
        part = view[i:i + chunk]
        part.copy_(torch.poisson(lam.expand(part.shape[0], 3, V), generator=gen))


def _members(c, seed):
    specs = [replace(r.tissue, seed=1 + seed) for r in W.batch(c["members"])]
    gen = torch.Generator(device="cuda").manual_seed(seed)
    # one allocation holds every member's state
    pool = torch.empty(sum(s.state_ints for s in specs), dtype=torch.int32, device="cuda")
    members, at = [], 0
    for s in specs:
        buf = pool[at:at + s.state_ints]
        at += s.state_ints
        members.append(Tissue(s, buffer=buf))
        _fill(buf, s.cells, s.V, (4.0 * s.model["kD"] + 3.0, 22.0, 4.0), gen)
    return specs, pool, members


def prepare(case, seed):
    c = dict(case)
    if c["kind"] == "serving":
        # requests of the serving workload that are all waiting (a request's
        # index is the seed of its tissues)
        c["reqs"] = [replace(r, index=(1 + seed) * 1000 + r.index, arrival_s=0.0,
                             replicas=min(r.replicas, c["replicas"]), side=min(r.side, 40),
                             n_steps=c["steps"], dt=c["dt"])
                     for r in W.serving(500)[c["first"]:c["first"] + c["requests"]]]
        return c
    if c["kind"] == "batch":
        specs, pool, members = _members(c, seed)
        torch.cuda.synchronize()
        c["batch"], c["tissues"], c["pool"] = Batch(members), members, pool
        if c["strang"]:
            c["batch"].set_splitting(SPLIT_STRANG)
        return c
    spec = _spec(c, seed)
    t = Tissue(spec)
    if c["strang"]:
        t.set_splitting(SPLIT_STRANG)
    gen = torch.Generator(device="cuda").manual_seed(seed)
    _fill(t.buffer, spec.cells, spec.V, _means(c), gen)
    c["tissue"] = t
    if c["io"]:
        c["host_in"] = torch.empty(spec.state_ints, dtype=torch.int32, pin_memory=True)
        c["host_in"].copy_(t.buffer)
        c["host_out"] = torch.empty_like(c["host_in"], pin_memory=True)
    return c


def run(state):
    if state["kind"] == "serving":
        server = Server(budget_bytes=8 << 30, chunk_steps=5, keep_counts=True)
        results = server.run(state["reqs"])
        # every replica's final counts, one array for the whole run
        return {"events": [r.events for r in results],
                "counts": np.concatenate([x for r in results for x in r.counts])}
    if state["kind"] == "batch":
        state["batch"].step(state["dt"], state["steps"])
        return {"counts": state["pool"]}
    t = state["tissue"]
    if state["io"]:
        t.write_counts_from(state["host_in"], step_index=0)
    t.step(state["dt"], state["steps"])
    out = {}
    if state["io"]:
        t.read_counts_into(state["host_out"])
        out["counts"] = state["host_out"]
    else:
        out["counts"] = t.buffer
    if state["stats"]:
        out["events"], out["t_last"] = t.read_stats()
    return out


def _hops(n):
    """Mean number of neighbour voxels."""
    return 4.0 * (n - 1) / n


def _cell_events(n, dt, means, kD=10.0):
    """Expected chi events of one Notch-Delta cell in a step: hops, decays and production."""
    D, N, R = means
    per_voxel = (D + N + R) * _hops(n) + 0.1 * (D + N) + 0.2 * R + kD / (1.0 + (R / 20.0) ** 2) + 5.0
    return n * n * dt * per_voxel


def _events(c):
    """Expected chi events of one pass."""
    if c["kind"] == "serving":
        # ~19x19 cells of 16x16 voxels per replica on average
        return c["requests"] * c["replicas"] * c["steps"] * 360.0 * _cell_events(16, c["dt"], START)
    if c["kind"] == "batch":
        return c["steps"] * sum(
            r.tissue.cells * _cell_events(r.tissue.n, c["dt"],
                                          (4.0 * r.tissue.model["kD"] + 3.0, 22.0, 4.0),
                                          r.tissue.model["kD"])
            for r in W.batch(c["members"]))
    cells = c["width"] * c["height"]
    if c["model"] == "promoter":
        n = c["n"]
        mols = 0.25 * n * n
        per_cell = c["dt"] * (mols * (n * n * _hops(n) + 1.0) + 100.0)
        inner = max(0, c["width"] - 2 * c["edge"]) * max(0, c["height"] - 2 * c["edge"])
        lattice = cells - (inner if c["edge"] >= 0 else 0)
        return c["steps"] * lattice * per_cell
    return c["steps"] * cells * _cell_events(c["n"], c["dt"], _means(c))


def _state_bytes(c):
    if c["kind"] == "serving":
        return 0.0  # states are made on the device and read back once: counted below
    if c["kind"] == "batch":
        return 4.0 * sum(r.tissue.state_ints for r in W.batch(c["members"]))
    return 12.0 * c["width"] * c["height"] * c["n"] ** 2


def work(case):
    """bytes: the state read and written once per pass.  flops: the integer
    operations of the events that the pass simulates, about 200 each: one
    Philox block (40 multiplications and as many logical operations), -ln u
    and one division in 64-bit integer arithmetic, and the selection."""
    c = dict(case)
    state = _state_bytes(c)
    if c["kind"] == "serving":
        state = 12.0 * c["requests"] * c["replicas"] * 360.0 * 256.0
    return {"bytes": 2.0 * state, "flops": 200.0 * _events(c)}


def exact(case, seed):
    """The outputs are whole numbers of one exact trajectory (and its event
    times): there is no value in real arithmetic to be near to."""
    return None
