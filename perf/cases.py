"""What users of this library have it do, as measurable cases: molecular dynamics on the device, evaluations for a driver that
owns the dynamics (on the device or on the host), screening of unrelated configurations, and neighbor-list export, from a few
hundred atoms to millions, in both precisions and with the options that production runs switch on.

The structures, species, temperatures and networks are those of `workloads` (a 6-species alloy, a unary metal, a 3-species
alloy, a 3-species ionic solid), here drawn on the GPU and for boxes of any number of cells per edge.  The networks are the
fixed ones of each workload (a user's model does not change from run to run); the configuration comes from the seed.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2608_16329_b200 as mlip
import workloads as wl

R_CUT, SKIN = 6.0, 1.0
DEVICE = 0

# Structure by name: workload number, lattice constant, sites per cell, displacement (Angstrom), mole fractions, temperature (K),
# time step (fs; the random networks have no repulsive core, so trajectories stay within a few fs of the lattice), and the
# fewest cells along an edge (a box edge holds two list radii).
STRUCTURES = {
    "hea6": dict(cfg=5, a=3.6, basis=wl._FCC_BASIS, sigma=0.05, fractions=[1.0 / 6.0] * 6, temperature=300.0, dt=1.0, least=4),
    "unary": dict(cfg=2, a=3.3, basis=wl._BCC_BASIS, sigma=0.08, fractions=[1.0], temperature=300.0, dt=1.0, least=5),
    "alloy3": dict(cfg=3, a=4.05, basis=wl._FCC_BASIS, sigma=0.05, fractions=[0.90, 0.05, 0.05], temperature=300.0, dt=1.0, least=4),
    "ionic3": dict(cfg=4, a=20.0 ** (1.0 / 3.0), basis=wl._SC_BASIS, sigma=0.10, fractions=[0.47, 0.12, 0.41], temperature=600.0, dt=0.4, least=6),
}


def _case(name, use, structure, cells, precision=0, k=32, l_max=3, steps=10, rebuild=10, deterministic=False, compact=False):
    """`use`: nve, nvt, evaluate, host, screen or lists (see `run`).  rebuild: list policy of the MD uses; of the host use, whether
    the call rebuilds the lists."""
    c = {"use": use, "structure": structure, "nx": cells[0], "ny": cells[1], "nz": cells[2], "precision": precision, "k": k, "l_max": l_max,
         "steps": steps if use in ("nve", "nvt") else 0, "rebuild": rebuild if use in ("nve", "nvt", "host") else 0,
         "deterministic": deterministic, "compact": compact}
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # one small periodic cell with new atoms in each call: active learning and dataset screening, a few hundred atoms each
        _case("screen 256", "screen", "hea6", (4, 4, 4)),
        # a small MD run on the device: ten NVE steps with the fixed rebuild interval
        _case("nve 864", "nve", "hea6", (6, 6, 6)),
        # the paper's ensemble (NVT at 300 K, rebuild on displacement checked every five steps) on a small pure metal
        _case("nvt 4394", "nvt", "unary", (13, 13, 13), steps=20, rebuild=-5),
        # one step of a driver that integrates the atoms itself with device tensors (a Python MD or relaxation loop)
        _case("evaluate 5544", "evaluate", "alloy3", (9, 11, 14)),
        # a reproducible run: integer accumulation of forces, energy and virial
        _case("nve 19652 reproducible", "nve", "hea6", (17, 17, 17), deterministic=True),
        # an ordinary run of a pure metal (the unary workload's own size)
        _case("nve 65536", "nve", "unary", (32, 32, 32)),
        # the double-precision path at an ordinary size
        _case("nve 55296 f64", "nve", "hea6", (24, 24, 24), precision=1),
        # the wider radial basis of the paper's ablation (double precision), configurations evaluated one by one
        _case("screen 6912 f64 k64", "screen", "hea6", (12, 12, 12), precision=1, k=64),
        # neighbor lists for analysis: build and export in canonical form
        _case("lists 108000", "lists", "hea6", (30, 30, 30)),
        # the call a host-side MD code makes per step: positions in, energy, forces and virial out (3-species workload's size)
        _case("host 1048576", "host", "alloy3", (64, 64, 64), rebuild=0),
        # a large run with compact (16-bit) neighbor lists, the memory-saving format (ionic workload's size)
        _case("nve 2000000 compact", "nve", "ionic3", (125, 125, 128), compact=True),
        # the benchmark size: ten NVE steps of 8 M atoms with one rebuild
        _case("nve 8001504", "nve", "hea6", (126, 126, 126)),
    ]


def draw(rng):
    use = rng.choice(["nve", "nve", "nve", "nvt", "evaluate", "host", "screen", "lists"])
    structure = rng.choice(["hea6", "hea6", "unary", "alloy3", "ionic3"])
    precision = 1 if use != "lists" and rng.random() < 0.25 else 0
    k, l_max = (rng.choice([16, 32, 32, 64]), rng.choice([2, 3, 3])) if precision else (32, 3)
    most = 250_000 if precision or use == "lists" else 2_000_000
    s = STRUCTURES[structure]
    atoms = math.exp(rng.uniform(math.log(256), math.log(most)))
    edge = (atoms / len(s["basis"])) ** (1.0 / 3.0)
    cells = tuple(max(s["least"], int(round(edge * math.exp(rng.uniform(-0.25, 0.25))))) for _ in range(3))
    steps = rng.choice([5, 10, 20]) if atoms < 100_000 else rng.choice([3, 5, 10])
    rebuild = rng.choice([10, 10, 5, -5]) if use in ("nve", "nvt") else int(rng.random() < 0.3)
    return _case(None, use, structure, cells, precision, k, l_max, steps, rebuild,
                 deterministic=precision == 0 and use == "nve" and rng.random() < 0.2, compact=rng.random() < 0.2)


def _atoms(case):
    return case["nx"] * case["ny"] * case["nz"] * len(STRUCTURES[case["structure"]]["basis"])


def _within(case, radius):
    """Mean number of atoms inside `radius` of an atom."""
    s = STRUCTURES[case["structure"]]
    return len(s["basis"]) / s["a"] ** 3 * 4.0 / 3.0 * math.pi * radius ** 3


def _configuration(case, seed):
    """Positions (inside the box), species, velocities and box edges of the case's structure, drawn on the GPU."""
    s = STRUCTURES[case["structure"]]
    dev = torch.device("cuda", DEVICE)
    gen = torch.Generator(device=dev)
    gen.manual_seed(int(seed) * 7919 + _atoms(case))
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    n = _atoms(case)
    cell = torch.arange(nx * ny * nz, device=dev)
    origin = torch.stack([cell // (ny * nz), cell // nz % ny, cell % nz], dim=1).to(torch.float64)
    pos = ((origin[:, None, :] + torch.as_tensor(s["basis"], device=dev)[None, :, :]) * s["a"]).reshape(n, 3)
    pos += s["sigma"] * torch.randn(n, 3, generator=gen, device=dev, dtype=torch.float64)
    box = np.array([nx, ny, nz], dtype=np.float64) * s["a"]
    edges = torch.as_tensor(box, device=dev)
    pos -= torch.floor(pos / edges) * edges
    pos[pos >= edges] = 0.0   # x = L after rounding belongs at 0
    mix = torch.tensor(s["fractions"], device=dev, dtype=torch.float64)
    species = torch.searchsorted(torch.cumsum(mix, 0), torch.rand(n, generator=gen, device=dev, dtype=torch.float64)).clamp_(max=len(mix) - 1).to(torch.int32)
    mass = torch.as_tensor(np.array(wl.MASSES[s["cfg"]]), device=dev, dtype=torch.float64)[species.long()]
    vel = torch.randn(n, 3, generator=gen, device=dev, dtype=torch.float64) * torch.sqrt(wl.KB_EV_PER_K * s["temperature"] * wl.ACC_UNIT / mass)[:, None]
    vel -= (mass[:, None] * vel).sum(dim=0) / mass.sum()
    return pos.contiguous(), species, vel.contiguous(), box


def prepare(case, seed):
    """The model's context, the configuration and (but for the uses that build them in each call) its neighbor lists."""
    s = STRUCTURES[case["structure"]]
    n_species = len(s["fractions"])
    cfg = s["cfg"]
    enc, head = wl.make_weights(n_species, wl.BASE_SEED + cfg + 1000, wl.ENC_OUT_SCALE[cfg], wl.HEAD_OUT_SCALE[cfg], k=case["k"], l_max=case["l_max"])
    pot = mlip.Potential(n_species, R_CUT, SKIN, enc, head, np.array(wl.MASSES[cfg]), device=DEVICE, precision=case["precision"], k=case["k"],
                         l_max=case["l_max"], force_mode=int(case["deterministic"]), list_format=int(case["compact"]))
    pos, species, vel, box = _configuration(case, seed)
    state = {"case": case, "pot": pot, "pos": pos, "species": species, "vel": vel, "box": box, "dt": s["dt"], "temperature": s["temperature"]}
    if case["use"] == "host":   # a host code's own arrays (page-locked, as an MD code that talks to a GPU keeps them)
        state["pos"] = pos.cpu().pin_memory()
        state["species"] = species.cpu().pin_memory()
        state["forces"] = torch.empty(pos.shape, dtype=torch.float32).pin_memory()
        mlip.mlip_compute_host(pot.ctx, state["pos"], state["species"], box, True, state["forces"])
    elif case["use"] == "lists":
        state["segments"] = torch.zeros(pos.shape[0] * n_species + 1, dtype=torch.int64, device=pos.device)
        state["neighbors"] = torch.zeros(int(1.5 * pos.shape[0] * _within(case, R_CUT + SKIN)), dtype=torch.int32, device=pos.device)
    elif case["use"] != "screen":
        pot.build_neighbors(pos, species, box)
    return state


def run(state):
    case, pot = state["case"], state["pot"]
    use = case["use"]
    if use in ("nve", "nvt"):   # a segment of a run from a given state: positions and velocities in, positions, velocities and energies out
        pot.set_state(pos=state["pos"], vel=state["vel"], step=0)
        if use == "nve":
            pot.step(case["steps"], state["dt"], case["rebuild"])
        else:
            mlip.mlip_reset_thermostat(pot.ctx)
            pot.step_nvt(case["steps"], state["dt"], case["rebuild"], state["temperature"])
        pos, vel, _ = pot.state()
        return {"pos": pos, "vel": vel, "energies": pot.energies()}
    if use == "evaluate":       # new positions, same lists
        pot.set_positions(state["pos"])
        return pot.compute()
    if use == "screen":         # a configuration of its own: lists and evaluation
        pot.build_neighbors(state["pos"], state["species"], state["box"])
        return pot.compute(want_e_atom=True)
    if use == "lists":          # build, then the canonical lists into the analysis code's own arrays
        pot.build_neighbors(state["pos"], state["species"], state["box"])
        _, total = mlip.mlip_get_neighbors(pot.ctx, state["segments"], state["neighbors"])
        return {"entries": total, "segments": state["segments"], "neighbors": state["neighbors"]}
    virial = np.empty(9)
    energy = mlip.mlip_compute_host(pot.ctx, state["pos"], state["species"], state["box"], bool(case["rebuild"]), state["forces"], virial)
    return {"energy": energy, "forces": state["forces"], "virial": virial}


def work(case):
    """Operations of the evaluations (pairs inside the cutoff and per-atom networks, FMA = 2; list tests for the uses that build) and
    the bytes of a pass's inputs and outputs."""
    s = STRUCTURES[case["structure"]]
    n = _atoms(case)
    pairs, entries = _within(case, R_CUT), _within(case, R_CUT + SKIN)
    k, d, n_inv = case["k"], (case["l_max"] + 1) ** 2, (case["l_max"] + 1) * case["k"]
    per_pair = 60 + 150 * d / 16 + 512 * k / 32 + 6 * d * k + 168 * d / 16     # geometry, harmonics, radial functions, contractions, projection
    per_atom = 3 * d * k + 4 * (n_inv * 64 + 3 * 64 * 64) + 256 + 5000         # invariants, network forward and reverse
    evaluation = pairs * per_pair + per_atom
    real = 8 if case["precision"] else 4
    use = case["use"]
    if use == "lists":
        return {"bytes": n * (24 + 4 + 4 * entries + 8 * len(s["fractions"])), "flops": n * entries * 8}
    if use in ("nve", "nvt"):
        return {"bytes": n * (48 + 48), "flops": n * evaluation * (case["steps"] + 1)}
    if use == "screen":
        return {"bytes": n * (24 + 4 + 4 * real), "flops": n * (evaluation + entries * 8)}
    return {"bytes": n * (24 + 3 * real), "flops": n * evaluation}


# Four times the largest difference seen over the listed and two dozen drawn cases: single precision against the double-precision
# path on the same inputs (forces rel 4.2e-6, max 2.1e-5; a trajectory's velocities rel 1.4e-6, max 6.8e-6), double precision against
# itself with twice the radial-table knots (forces rel 5.6e-10, max 1.9e-9; velocities rel 4.4e-11, max 6.9e-10).
TOLERANCE = {
    ("evaluation", 0): {"rel": 1.7e-5, "max": 8.6e-5}, ("trajectory", 0): {"rel": 5.6e-6, "max": 2.8e-5},
    ("evaluation", 1): {"rel": 2.3e-9, "max": 7.6e-9}, ("trajectory", 1): {"rel": 1.8e-10, "max": 2.8e-9},
}


def tolerance(case):
    if case["use"] == "lists":
        return "exact"
    return TOLERANCE["trajectory" if case["use"] in ("nve", "nvt") else "evaluation", case["precision"]]
