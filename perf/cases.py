"""The work a user of the library has it do, as timed cases.

Every case goes through the package's public classes (``Lattice``, ``Batch``)
with their automatic settings, on inputs that ``prepare`` makes on the device
from a seed.  A case's ``kind`` says which calls one pass makes:

  * ``run``     advance one lattice, then take a snapshot: its coarse-grained
                fields (where the block divides the sides) and its node bytes;
  * ``batch``   advance many lattices together, then read every member's
                coarse-grained fields back to the host;
  * ``resume``  load node bytes, advance a few steps, store node bytes;
  * ``coarse``  coarse-grain a lattice that rests on the device;
  * ``setup``   start a run from nothing: obstacles from shapes, a generated
                initial state, and its node bytes.

Sizes, densities, forcing probabilities and obstacles are those of the
repository's workloads (``workloads.py``), its tests and its serving trace.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

import paper_1208_2428_gb300 as fhp

# Word operations per 32 nodes and step: scattering, one-node shifts, and one
# Philox4x32-10 block per four words (two with forcing).
_OPS_PER_WORD_STEP = 100.0


def listed():
    return [
        # A small periodic box, the study of a single relaxation: the step loop is all latency.
        {"name": "run_periodic_256", "kind": "run", "W": 256, "H": 256, "steps": 100, "density": 0.3, "p": 0.0,
         "obstacle": "none", "rules": 2, "block": 32},
        # The channel workload: forced flow between walls, fields taken every 1,000 steps.
        {"name": "run_channel_4096x1024", "kind": "run", "W": 4096, "H": 1024, "steps": 1000, "density": 0.2,
         "p": 1e-3, "obstacle": "walls", "rules": 2, "block": 32},
        # The benchmark's cylinder: the largest lattice that about fits L2.
        {"name": "run_cylinder_16384x4096", "kind": "run", "W": 16384, "H": 4096, "steps": 200, "density": 0.25,
         "p": 5e-4, "obstacle": "cylinder", "rules": 2, "block": 32},
        # The paper's GPU lattice: far beyond L2, the width not a whole number of 128-node quads.
        {"name": "run_paper_29984x27990", "kind": "run", "W": 29984, "H": 27990, "steps": 20, "density": 0.25,
         "p": 5e-4, "obstacle": "cylinder", "rules": 2, "block": 0},
        # A porous medium on odd sizes, FHP-I, pushed hard (every warp meets forced nodes).
        {"name": "run_porous_3104x1498", "kind": "run", "W": 3104, "H": 1498, "steps": 200, "density": 0.35,
         "p": 0.02, "obstacle": "points", "rules": 1, "block": 0},
        # The collision-saturated rules on a mid-sized cylinder.
        {"name": "run_fhp3_4096x2048", "kind": "run", "W": 4096, "H": 2048, "steps": 200, "density": 0.25,
         "p": 5e-4, "obstacle": "cylinder", "rules": 3, "block": 32},
        # An ensemble average: many mid-sized porous lattices for a long time in one call.
        {"name": "batch_ensemble_64", "kind": "batch", "count": 64, "lo": 128, "hi": 2048, "law": "uniform",
         "steps": 1000, "quantum": 1000, "p": 0.0, "obstacle": "points"},
        # What the serving loop does: mixed sizes, half of them cylinders, in quanta of 64 steps.
        {"name": "batch_serving_24", "kind": "batch", "count": 24, "lo": 256, "hi": 8192, "law": "log",
         "steps": 256, "quantum": 64, "p": 5e-4, "obstacle": "cylinder"},
        # A parameter sweep over small boxes in short calls: launches and hand-offs count.
        {"name": "batch_sweep_16", "kind": "batch", "count": 16, "lo": 128, "hi": 512, "law": "uniform",
         "steps": 96, "quantum": 32, "p": 0.0, "obstacle": "none"},
        # Restart from a checkpoint, a few steps on, and the next checkpoint.
        {"name": "resume_8192x4096", "kind": "resume", "W": 8192, "H": 4096, "steps": 8, "density": 0.25,
         "p": 5e-4, "obstacle": "cylinder", "rules": 2},
        # Fields of a resting lattice, for a plot or a check of convergence.
        {"name": "coarse_16384x4096", "kind": "coarse", "W": 16384, "H": 4096, "density": 0.25,
         "obstacle": "cylinder", "block": 64},
        # A new request: obstacles and initial state made on the device, first snapshot.
        {"name": "setup_4096x4096", "kind": "setup", "W": 4096, "H": 4096, "density": 0.3,
         "obstacle": "cylinder"},
    ]


def _log_int(rng, lo, hi, mult):
    v = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return max(lo, min(hi, int(round(v / mult)) * mult))


def draw(rng: random.Random):
    kind = rng.choice(["run", "run", "run", "run", "batch", "batch", "resume", "coarse", "setup"])
    obstacle = rng.choice(["none", "walls", "cylinder", "points"])
    p = rng.choice([0.0, 5e-4, 1e-3, 0.02])
    density = round(rng.uniform(0.1, 0.5), 3)
    if kind == "batch":
        law = rng.choice(["uniform", "log"])
        hi = rng.choice([512, 1024, 2048])
        steps = _log_int(rng, 32, 1000, 1)
        return {"kind": kind, "count": _log_int(rng, 4, 64, 1), "lo": rng.choice([128, 256]), "hi": hi, "law": law,
                "steps": steps, "quantum": rng.choice([steps, min(steps, 64)]), "p": p, "obstacle": obstacle}
    if kind == "coarse":
        block = rng.choice([32, 64, 96, 128])
        return {"kind": kind, "W": _log_int(rng, 512 // block * block, 16384 // block * block, block),
                "H": _log_int(rng, 512 // block * block, 4096 // block * block, 2 * block), "density": density,
                "obstacle": obstacle, "block": block}
    W, H = _log_int(rng, 256, 16384, 32), _log_int(rng, 128, 8192, 2)
    if kind == "setup":
        return {"kind": kind, "W": W, "H": H, "density": density, "obstacle": obstacle}
    rules = rng.choice([2, 2, 2, 1, 3])
    if kind == "resume":
        return {"kind": kind, "W": W, "H": H, "steps": rng.randint(1, 16), "density": density, "p": p,
                "obstacle": obstacle, "rules": rules}
    # As many steps as keep the pass within the cylinder workload's 200 steps.
    most = max(20, min(1000, int(16384 * 4096 * 200 / (W * H) / (3 if rules == 3 else 1))))
    return {"kind": kind, "W": W, "H": H, "steps": _log_int(rng, 20, most, 1), "density": density, "p": p,
            "obstacle": obstacle, "rules": rules, "block": 32 if W % 32 == 0 and H % 32 == 0 else 0}


# -- inputs -----------------------------------------------------------------------
def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed) & 0x7FFFFFFF)


def _shapes(W, H, obstacle):
    walls = [(fhp.SHAPE_ROWS, 0, 1, 0), (fhp.SHAPE_ROWS, H - 1, H, 0)]
    if obstacle == "walls":
        return walls
    if obstacle == "cylinder":
        return walls + [(fhp.SHAPE_DISC, W // 4, H // 2, max(1, H // 16))]
    return []


def _solid(W, H, obstacle, gen):
    """The solid mask as a boolean device tensor (walls and the cylinder of
    ``_shapes``, or 1 % of the nodes at random)."""
    m = torch.zeros((H, W), dtype=torch.bool, device="cuda")
    if obstacle == "points":
        for y in range(0, H, 1024):
            m[y:y + 1024] = torch.rand(m[y:y + 1024].shape, device="cuda", generator=gen) < 0.01
    if obstacle in ("walls", "cylinder"):
        m[0] = True
        m[H - 1] = True
    if obstacle == "cylinder":
        yy = torch.arange(H, device="cuda")[:, None] - H // 2
        xx = torch.arange(W, device="cuda")[None, :] - W // 4
        m |= xx * xx + yy * yy <= max(1, H // 16) ** 2
    return m


def _node_bytes(case, seed):
    """H x W node bytes on the device: every mover and rest bit of a fluid
    node set with the case's density, solid nodes with bit 7 alone."""
    W, H = case["W"], case["H"]
    gen = _generator(seed)
    solid = _solid(W, H, case["obstacle"], gen)
    out = torch.empty((H, W), dtype=torch.uint8, device="cuda")
    for y in range(0, H, 1024):
        o = out[y:y + 1024]
        o.zero_()
        for bit in range(7):
            o |= (torch.rand(o.shape, device="cuda", generator=gen) < case["density"]).to(torch.uint8) << bit
        o[solid[y:y + 1024]] = 0x80
    return out


def _members(case, seed):
    """(W, H, density, p, obstacle) of a batch's members: the sizes belong to
    the case, the densities to the seed."""
    sizes, values = random.Random(4), random.Random(int(seed))
    lo, hi = case["lo"], case["hi"]
    out = []
    for i in range(case["count"]):
        if case["law"] == "log":
            W, H = _log_int(sizes, lo, hi, 64), _log_int(sizes, lo, hi, 64)
        else:
            W, H = (lo + 64 * sizes.randrange((hi - lo) // 64 + 1) for _ in range(2))
        plain = case["obstacle"] == "cylinder" and i % 2 == 1
        out.append((W, H, values.uniform(0.1, 0.4), 0.0 if plain else case["p"],
                    "none" if plain else case["obstacle"]))
    return out


def prepare(case, seed):
    kind = case["kind"]
    state = {"case": case}
    if kind == "batch":
        members = _members(case, seed)
        batch = fhp.Batch(sum(fhp.Batch.lattice_bytes(m[0], m[1]) for m in members) + (64 << 20))
        gen = _generator(seed)
        slots, masks = [], []
        for i, (W, H, density, p, obstacle) in enumerate(members):
            slot = batch.add(W, H, int(seed) * 1000 + i, p)
            if obstacle == "points":
                masks.append(_solid(W, H, obstacle, gen).to(torch.uint8).cpu().numpy())
                batch.load_obstacles(slot, masks[-1])
            elif obstacle != "none":
                batch.load_obstacle_shapes(slot, _shapes(W, H, obstacle))
            batch.init_random(slot, density)
            slots.append(slot)
        batch.synchronize()
        state.update(batch=batch, slots=slots, masks=masks)
        return state
    W, H = case["W"], case["H"]
    lat = fhp.Lattice(W, H, seed=int(seed), forcing_p=case.get("p", 0.0))
    lat.set_rules(case.get("rules", 2))
    state["lattice"] = lat
    if kind == "coarse":
        lat.set_state_tensor(_node_bytes(case, seed))
    elif kind == "resume":
        state["input"] = _node_bytes(case, seed)
    elif kind == "run":
        if case["obstacle"] == "points":
            state["mask"] = _solid(W, H, "points", _generator(seed)).to(torch.uint8).cpu().numpy()
            lat.load_obstacles(state["mask"])
        else:
            lat.load_obstacle_shapes(_shapes(W, H, case["obstacle"]))
        lat.init_random(case["density"])
    if kind != "coarse":
        state["bytes"] = torch.empty((H, W), dtype=torch.uint8, device="cuda")
    B = case.get("block", 0)
    if B:
        state["counts"] = torch.empty((H // B, W // B, 9), dtype=torch.int32, device="cuda")
        state["fields"] = [torch.empty((H // B, W // B), dtype=torch.float32, device="cuda") for _ in range(3)]
    lat.synchronize()
    return state


# -- one pass ---------------------------------------------------------------------
def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "batch":
        batch = state["batch"]
        left = case["steps"]
        while left > 0:
            n = min(left, case["quantum"])
            batch.step(n)
            left -= n
        done = torch.cuda.Event()
        done.record(batch.stream)
        handles = [batch.coarse_grain_begin(slot, 32, done) for slot in state["slots"]]
        got = [batch.coarse_grain_finish(h) for h in handles]
        return [np.concatenate([g[k].reshape(-1) for g in got]) for k in range(4)]
    lat = state["lattice"]
    if kind == "coarse":
        lat.coarse_grain_into(case["block"], state["counts"], *state["fields"])
        return [state["counts"], *state["fields"]]
    if kind == "setup":
        lat.load_obstacle_shapes(_shapes(case["W"], case["H"], case["obstacle"]))
        lat.init_random(case["density"])
        return lat.get_state_tensor(out=state["bytes"])
    if kind == "resume":
        lat.set_state_tensor(state["input"])
        lat.step(case["steps"])
        return lat.get_state_tensor(out=state["bytes"])
    lat.step(case["steps"])
    out = [lat.get_state_tensor(out=state["bytes"])]
    if case["block"]:
        lat.coarse_grain_into(case["block"], state["counts"], *state["fields"])
        out += [state["counts"], *state["fields"]]
    return out


# -- what a pass cannot do without ------------------------------------------------
def work(case):
    kind = case["kind"]
    if kind == "batch":
        nodes = sum(W * H for W, H, *_ in _members(case, 0))
        # The members' planes in (8 bits a node) and out (7), the fields out.
        return {"bytes": nodes * (15 / 8) + nodes / 1024 * 48,
                "flops": nodes / 32 * case["steps"] * _OPS_PER_WORD_STEP}
    nodes = case["W"] * case["H"]
    if kind == "coarse":
        return {"bytes": nodes + nodes / case["block"] ** 2 * 48, "flops": nodes / 32 * 15}
    if kind == "setup":
        # Out: 8 planes and the node bytes; 28 Philox blocks per 32 nodes.
        return {"bytes": nodes * 2.0, "flops": nodes / 32 * 28 * 60.0}
    fields = nodes / case["block"] ** 2 * 48 if case.get("block") else 0
    if kind == "resume":
        return {"bytes": nodes * (1 + 1 + 15 / 8), "flops": nodes / 32 * case["steps"] * _OPS_PER_WORD_STEP}
    return {"bytes": nodes * (15 / 8 + 1) + fields, "flops": nodes / 32 * case["steps"] * _OPS_PER_WORD_STEP}


# -- the same in 64 bits -----------------------------------------------------------
def exact(case, seed):
    """Coarse-grained fields of given node bytes in 64-bit arithmetic.  (The
    other cases' floating outputs are derived from evolved lattices, whose
    bits have no shorter description than the automaton itself.)"""
    if case["kind"] != "coarse":
        return None
    B, W, H = case["block"], case["W"], case["H"]
    nodes = _node_bytes(case, seed)
    fluid = (nodes & 0x80) == 0

    def block_sum(mask):
        return mask.view(H // B, B, W // B, B).sum(dim=(1, 3), dtype=torch.float64)

    n = [block_sum(((nodes >> i) & 1).bool() & fluid) for i in range(7)]
    f = block_sum(fluid)
    mass = sum(n)
    jx = -n[0] + n[1] + 2 * n[2] + n[3] - n[4] - 2 * n[5]
    jy = -n[0] - n[1] + n[3] + n[4]
    zero = torch.zeros_like(f)
    rho = torch.where(f > 0, mass / f.clamp(min=1), zero)
    ux = torch.where(mass > 0, jx / (2 * mass.clamp(min=1)), zero)
    uy = torch.where(mass > 0, math.sqrt(3) / 2 * jy / mass.clamp(min=1), zero)
    counts = torch.stack(n + [f, mass], dim=-1).to(torch.int32)
    return [counts, rho, ux, uy]
