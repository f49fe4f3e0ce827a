"""Cases of the energy / force / virial path and of its molecular dynamics drivers, over the sizes,
models and options in which the library is used.

A case names a model (a workload of ``workloads.configs``: widths, stored calibration, head scale;
the weights are a user's fixed model, the atoms come from the seed), a structure and a pass:

  point   energy, forces, virial and atomic energies of positions on a list that is kept: what a
          relaxation or an external integrator calls in its loop
  fresh   the list is built, then evaluated: the first call on a new structure
  energy  the list is built, then energies alone: screening, Monte Carlo
  batch   many independent frames of unequal size in one call: evaluation of a data set
  nve     a snapshot is copied in, the list built, and the velocity Verlet driver run with a rebuild
          every ten steps (it evaluates once for the opening kick and once per step); the segment
          ends with the frame that a trajectory keeps: energy, forces, virial, atomic energies
  nvt     the same under the thermostat

Structures are jittered lattices with randomly left out sites, so that any number of atoms can be
had: densities, jitters and cell edges are those of the workloads.
"""

import math

import numpy as np
import torch

from paper_2608_19041_b200 import binding
from workloads import CONFIGS, workload_blob, workload_profile

SKIN = 1.0
KB = 8.617333262e-5          # eV / K
ACCEL = 9648.53321           # (eV / Angstrom / amu) in Angstrom / ps^2

# lattice: sites per cell, cell edge, jitter (normal, or uniform where the minimum distance matters)
LATTICES = {
    "fcc_al": dict(basis="fcc", a=4.05, normal=0.05),
    "fcc_cu": dict(basis="fcc", a=3.615, normal=0.1),
    "bcc": dict(basis="bcc", a=3.2, normal=0.08),
    "diamond": dict(basis="diamond", a=3.567, normal=0.03),
    # 0.08 atoms per cubic Angstrom, no two closer than 1.8 Angstrom
    "amorphous": dict(basis="sc", a=0.08 ** (-1.0 / 3.0), uniform=0.26),
    # molecules at 1.0 g/cm^3 (29.92 cubic Angstrom each), oxygens no closer than 2.5 Angstrom
    "water": dict(basis="sc", a=29.92 ** (1.0 / 3.0), uniform=0.3),
}
BASES = {
    "sc": [[0, 0, 0]],
    "bcc": [[0, 0, 0], [.5, .5, .5]],
    "fcc": [[0, 0, 0], [.5, .5, 0], [.5, 0, .5], [0, .5, .5]],
    "diamond": [[0, 0, 0], [.5, .5, 0], [.5, 0, .5], [0, .5, .5],
                [.25, .25, .25], [.75, .75, .25], [.75, .25, .75], [.25, .75, .75]],
}
LATTICE_OF = {"cfg1_al108": "fcc_al", "cfg2_cu4000": "fcc_cu", "cfg3_water32400": "water", "cfg4_hea128k": "bcc",
              "cfg5_amorphous1m": "amorphous", "paper_nano_c1m": "diamond", "paper_mini_c1m": "diamond",
              "paper_neo_c1m": "diamond", "paper_air_c1m": "diamond", "paper_plus_c1m": "diamond"}


def _case(name, kind, model, atoms, modes=0, frames=0, steps=0, sheared=False, slab=False, ghosts=False):
    c = {"pass": kind, "model": model, "atoms": atoms, "modes": modes, "frames": frames, "steps": steps,
         "sheared": sheared, "slab": slab, "ghosts": ghosts}
    return dict(c, name=name) if name else c


def listed():
    return [
        # a calculator inside a relaxation of the smallest benchmark cell: launches and latency
        _case("al_108_point", "point", "cfg1_al108", 108),
        # a new small molecular box, as an active-learning loop or a script meets one after another
        _case("water_597_fresh", "fresh", "cfg3_water32400", 597),
        # validation of a data set: 64 cells of 54 to 108 atoms per call
        _case("al_batch_64", "batch", "cfg1_al108", 108, frames=64),
        # classical MD of a few thousand atoms, one species: the latency-bound middle
        _case("cu_4000_nve", "nve", "cfg2_cu4000", 4000, steps=50),
        # water box, two species, degree three
        _case("water_32400_nve", "nve", "cfg3_water32400", 32400, steps=20),
        # five-component alloy, C0 = 128, under the thermostat; an odd number of atoms
        _case("alloy_127993_nvt", "nvt", "cfg4_hea128k", 127993, steps=10),
        # screening of a strained alloy cell: general cell, energies only (no backward pass)
        _case("alloy_30011_energy", "energy", "cfg4_hea128k", 30011, sheared=True),
        # the largest single-GPU workload: a million atoms of 64 species
        _case("amorphous_1m_nve", "nve", "cfg5_amorphous1m", 1000000, steps=10),
        # the same mixture with four shared radial modes (every edge reads its pair's mode mixing)
        _case("amorphous_modes4_40009_point", "point", "cfg5_amorphous1m", 40009, modes=4),
        # one spatial domain of a distributed run: owned atoms and ghosts around them, open box
        _case("amorphous_brick_8000_point", "point", "cfg5_amorphous1m", 8000, ghosts=True),
        # the narrowest and the widest of the published model variants on dense carbon (158 neighbours)
        _case("carbon_nano_216000_nvt", "nvt", "paper_nano_c1m", 216000, steps=10),
        _case("carbon_plus_64007_slab", "fresh", "paper_plus_c1m", 64007, slab=True),
    ]


def draw(rng):
    def atoms(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    model = rng.choice(["cfg1_al108", "cfg2_cu4000", "cfg3_water32400", "cfg4_hea128k", "cfg5_amorphous1m", "cfg5_amorphous1m",
                        "paper_nano_c1m", "paper_mini_c1m", "paper_neo_c1m", "paper_air_c1m"])
    kind = rng.choice(["point", "fresh", "energy", "batch", "nve", "nvt"])
    modes = 4 if model == "cfg5_amorphous1m" and rng.random() < 0.3 else 0
    if kind == "batch":
        return _case(None, kind, model, atoms(32, 400), modes=modes, frames=atoms(2, 128))
    if kind in ("nve", "nvt"):
        n = atoms(256, 250000)
        return _case(None, kind, model, n, modes=modes, steps=10 if n > 20000 else 40)
    ghosts = kind == "point" and rng.random() < 0.25
    sheared = not ghosts and rng.random() < 0.25
    slab = not ghosts and not sheared and rng.random() < 0.25
    return _case(None, kind, model, atoms(64, 300000), modes=modes, sheared=sheared, slab=slab, ghosts=ghosts)


def _grid(cells):
    """Edges of the most cube-like grid among those that exceed ``cells`` least."""
    side = max(1, int(round(cells ** (1.0 / 3.0))))
    span = range(max(1, side - 2), side + 3)
    return min(((nx, ny, -(-cells // (nx * ny))) for nx in span for ny in span),
               key=lambda g: g[0] * g[1] * g[2] - cells + (max(g) - min(g)) * cells / 10.0)


def _structure(case, atoms, gen):
    """(pos [N,3] float64, types [N] int32, cell [3,3] numpy) on the GPU."""
    lat = LATTICES[LATTICE_OF[case["model"]]]
    cfg = CONFIGS[case["model"]]["system"]
    water = cfg["kind"] == "water"
    sites = max(1, atoms // 3) if water else atoms
    basis = torch.tensor(BASES[lat["basis"]], dtype=torch.float64, device="cuda")
    n = _grid(-(-sites // len(basis)))
    axes = [torch.arange(k, dtype=torch.float64, device="cuda") for k in n]
    origin = torch.stack(torch.meshgrid(*axes, indexing="ij"), dim=-1).reshape(-1, 1, 3)
    pos = (origin + basis).reshape(-1, 3) * lat["a"]
    keep = torch.randperm(len(pos), generator=gen, device="cuda")[:sites]
    pos = pos[keep.sort().values]
    if "normal" in lat:
        pos = pos + lat["normal"] * torch.randn(pos.shape, generator=gen, dtype=torch.float64, device="cuda")
    else:
        pos = pos + lat["uniform"] * (2.0 * torch.rand(pos.shape, generator=gen, dtype=torch.float64, device="cuda") - 1.0)
    if water:       # rigid molecules, uniformly random orientations
        q = torch.randn((sites, 4), generator=gen, dtype=torch.float64, device="cuda")
        w, x, y, z = (q / q.norm(dim=1, keepdim=True)).unbind(1)
        ex = torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y + z * w), 2 * (x * z - y * w)], dim=1)
        ez = torch.stack([2 * (x * z + y * w), 2 * (y * z - x * w), 1 - 2 * (x * x + y * y)], dim=1)
        half = math.radians(104.5) / 2.0
        hx, hz = 0.96 * math.sin(half), 0.96 * math.cos(half)
        pos = torch.stack([pos, pos + hx * ex + hz * ez, pos - hx * ex + hz * ez], dim=1).reshape(-1, 3)
        types = torch.tensor([0, 1, 1], dtype=torch.int32, device="cuda").repeat(sites)
    elif "type_index" in cfg:
        types = torch.full((sites,), cfg["type_index"], dtype=torch.int32, device="cuda")
    else:
        types = torch.randint(0, cfg["n_types"], (sites,), generator=gen, dtype=torch.int32, device="cuda")
    cell = np.diag([k * lat["a"] for k in n]).astype(np.float64)
    if case["sheared"]:
        strain = np.array([[1.0, 0.0, 0.0], [0.12, 1.0, 0.0], [0.07, -0.05, 1.0]])
        cell = cell @ strain
        pos = pos @ torch.as_tensor(strain, device="cuda")
    return pos.contiguous(), types.contiguous(), cell


def _with_ghosts(pos, types, cell, reach):
    """The box's own atoms, then their periodic copies within about ``reach`` of it, nearest first (as
    one rank of a spatial decomposition holds them): as many as that shell holds on average."""
    edge = torch.as_tensor(np.diag(cell).copy(), device="cuda")
    pos = pos - torch.floor(pos / edge) * edge
    grown = [e + 2.0 * reach for e in edge.tolist()]
    count = int(len(pos) * (math.prod(grown) / math.prod(edge.tolist()) - 1.0))
    rep = [int(math.ceil((reach + 2.0) / e)) for e in edge.tolist()]
    images = [(x, y, z) for x in range(-rep[0], rep[0] + 1) for y in range(-rep[1], rep[1] + 1)
              for z in range(-rep[2], rep[2] + 1) if (x, y, z) != (0, 0, 0)]
    shift = torch.tensor(images, dtype=torch.float64, device="cuda") * edge
    copies = (pos.unsqueeze(0) + shift.unsqueeze(1)).reshape(-1, 3)
    outside = torch.maximum(-copies, copies - edge).amax(dim=1)
    near = torch.argsort(outside)[:count]
    return torch.cat([pos, copies[near]]).contiguous(), torch.cat([types, types.repeat(len(images))[near]]).contiguous()


def _velocities(types, masses, temperature, gen):
    m = torch.as_tensor(masses, device="cuda")[types.long()].unsqueeze(1)
    v = torch.randn((len(types), 3), generator=gen, dtype=torch.float64, device="cuda") * torch.sqrt(KB * temperature * ACCEL / m)
    return (v - (m * v).sum(dim=0) / m.sum()).contiguous()


def _model(case):
    return binding.Model(workload_blob(case["model"], case["modes"] or None))


def prepare(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    kind = case["pass"]
    s = {"case": case, "model": _model(case), "pbc": (1, 1, 0 if case["slab"] else 1)}
    if kind == "batch":
        # sizes between half of ``atoms`` and all of it, in no order
        low = -(-case["atoms"] // 2)
        frames = [_structure(case, low + (k * 37) % (case["atoms"] - low + 1), gen) for k in range(case["frames"])]
        s["offsets"] = np.cumsum([0] + [len(p) for p, _, _ in frames])
        s["pos"] = torch.cat([p for p, _, _ in frames]).contiguous()
        s["types"] = torch.cat([t for _, t, _ in frames]).contiguous()
        s["cells"] = np.stack([c for _, _, c in frames])
        return s
    pos, types, cell = _structure(case, case["atoms"], gen)
    if case["ghosts"]:
        owned = len(pos)
        pos, types = _with_ghosts(pos, types, cell, CONFIGS[case["model"]]["profile"]["rc"] + SKIN)
        s["pbc"] = (0, 0, 0)
        s["model"].set_owned_atoms(owned)
    s.update(pos=pos, types=types, cell=cell, forces=torch.empty_like(pos),
             energies=torch.empty(len(pos), dtype=torch.float64, device="cuda"))
    if kind == "point":
        s["model"].build_neighbors(pos, types, cell, s["pbc"], SKIN)
    elif kind in ("nve", "nvt"):
        md = CONFIGS[case["model"]]["md"] or dict(dt_ps=0.001, temperature=300.0)
        s["masses"] = CONFIGS[case["model"]]["system"]["masses"]
        s["dt"], s["temperature"] = md["dt_ps"], md["temperature"]
        s["vel"] = _velocities(types, s["masses"], md["temperature"], gen)
        s["work_pos"], s["work_vel"] = torch.empty_like(pos), torch.empty_like(pos)
    return s


def run(s):
    m, kind = s["model"], s["case"]["pass"]
    if kind == "batch":
        return m.compute_batch(s["offsets"], s["pos"], s["types"], s["cells"], s["pbc"], atom_energy=True)
    if kind == "energy":
        m.build_neighbors(s["pos"], s["types"], s["cell"], s["pbc"], 0.0)
        out = m.compute(s["pos"], forces=False, virial=False, out_atom_energy=s["energies"])
        return {"energy": out["energy"], "atom_energy": out["atom_energy"]}
    if kind in ("point", "fresh"):
        if kind == "fresh":
            m.build_neighbors(s["pos"], s["types"], s["cell"], s["pbc"], SKIN)
        return m.compute(s["pos"], out_forces=s["forces"], out_atom_energy=s["energies"])
    pos, vel = s["work_pos"], s["work_vel"]
    pos.copy_(s["pos"])
    vel.copy_(s["vel"])
    m.build_neighbors(pos, s["types"], s["cell"], s["pbc"], SKIN)
    m.set_md_state(pos, vel, s["masses"])
    if kind == "nve":
        e = m.step(s["case"]["steps"], s["dt"], rebuild_every=10)
    else:
        e = m.step_nvt(s["case"]["steps"], s["dt"], s["temperature"], 0.1, rebuild_every=10)
    out = m.compute(pos, out_forces=s["forces"], out_atom_energy=s["energies"])
    return dict(out, pos=pos, vel=vel, run=list(e))


def work(case):
    """Arithmetic of the model itself (one multiply-add is two): per edge inside the cutoff and per
    atom; bytes of the atoms' inputs and results, the model's constants read once per pass."""
    p = workload_profile(case["model"], case["modes"] or None)
    lat = LATTICES[LATTICE_OF[case["model"]]]
    water = CONFIGS[case["model"]]["system"]["kind"] == "water"
    density = len(BASES[lat["basis"]]) * (3 if water else 1) / lat["a"] ** 3
    atoms = case["atoms"] * (0.75 * case["frames"] if case["frames"] else 1)
    edges = atoms * density * 4.0 / 3.0 * math.pi * p["rc"] ** 3
    C0, R, S = p["C0"], p["R"], p["S"]
    forward = 6 * (C0 + R) + 2 * C0 * (1 + R) + 2 * S + C0 + p["C1"] + 60
    backward = 10 * (C0 + R) + 4 * C0 * (1 + R) + 4 * S + 2 * C0 + 250
    mlp = 2 * (p["D_out"] * p["F"] + (p["n_hidden"] - 1) * p["F"] ** 2 + p["F"])
    gradient = case["pass"] != "energy"
    evaluations = 1 + (case["steps"] + 1 if case["steps"] else 0)
    flops = evaluations * (edges * (forward + (backward if gradient else 0)) + atoms * mlp * (2 if gradient else 1))
    weights = 4 * (p["D_out"] * p["F"] + (p["n_hidden"] - 1) * p["F"] ** 2) + 12 * (C0 + R) * p["rc"] / p["table_dx"]
    # positions and species in, atomic energies out; forces out, or positions and velocities back
    per_atom = 28 + 8 + (24 if gradient else 0) + (48 if case["steps"] else 0)
    return {"bytes": atoms * per_atom + weights, "flops": flops}


def tolerance(case):
    """Largest relative differences, about four times what the library's other single-precision
    evaluations of the same model show against its default one (CUDA-core MLP, pair cache instead of
    per-pair tables, half the table spacing, smaller tiles): 4e-6 in the forces, virial and atomic
    energies.  The total energy of the 64-species model is a sum over atoms of both signs that
    cancels to a tenth of its terms and shows 2e-5."""
    return {"rel": 8e-5 if case["model"] == "cfg5_amorphous1m" else 1.6e-5}
