"""Shared radial modes by moments of the rows (many rows, no per-pair tables) against the same kernels reading every
edge's pair rows (few rows)."""

import numpy as np
import pytest
import torch

from oracle import dpa4c as orc
from workloads import SMALL_PROFILES, make_blob, make_system

pytestmark = pytest.mark.gpu

MOMENT_ROWS = 2048      # the fewest rows that take the way over moments


# one species (groups far from whole blocks of 64 rows come from the sizes), several, and more than the rows hold of
@pytest.mark.parametrize("species", [1, 3, 40])
@pytest.mark.parametrize("name", ["p32_2_4", "p32_3_2", "p32_4_2", "p64_3_8", "p128_3_4", "p128_4_4"])
def test_moments_match_modes_per_edge(name, species):
    from paper_2608_19041_b200 import binding
    p = dict(SMALL_PROFILES[name], T=species)
    masses = [1.0] * species
    dense = make_system(dict(kind="random_box", atoms=29, edges=(8.0, 8.5, 9.0), min_dist=1.6, seed=81, n_types=species, masses=masses))
    sparse = make_system(dict(kind="random_box", atoms=3, edges=(30.0, 30.0, 30.0), min_dist=1.6, seed=82, n_types=species, masses=masses))
    sparse["pos"][:2] = [[3.0, 3.0, 3.0], [4.7, 3.2, 3.1]]
    sizes, cells = (29, 3), [np.diag(np.diag(np.asarray(f["cell"], dtype=np.float64))) for f in (dense, sparse)]
    blob = make_blob(p, seed=83, bias_scale=0.2, e_ref_scale=0.5)
    m = binding.Model(blob, pair_table_mb=-1)
    tiled = binding.Model(blob, pair_table_mb=-1, node_tile=MOMENT_ROWS + 1)      # a tile by moments, one of 95 rows without

    def evaluate(model, copies):
        off = np.concatenate([[0], np.cumsum(np.tile(sizes, copies))])
        pos = np.tile(np.concatenate([dense["pos"], sparse["pos"]]), (copies, 1))
        types = np.tile(np.concatenate([dense["types"], sparse["types"]]), copies)
        out = model.compute_batch(off, torch.as_tensor(pos, dtype=torch.float64).cuda().contiguous(),
                                  torch.as_tensor(types, dtype=torch.int32).cuda().contiguous(),
                                  np.stack(cells * copies), (1, 1, 1), atom_energy=True)
        return (out["forces"].cpu().numpy().reshape(copies, 32, 3), out["atom_energy"].cpu().numpy().reshape(copies, 32),
                np.asarray(out["virials"]).reshape(copies, 2, -1))

    most = MOMENT_ROWS // 32
    Fb, Eb, Vb = evaluate(m, most - 1)       # every edge reads its pair's rows
    f_scale, e_scale = np.abs(Fb).max(), np.abs(Eb).max()
    by_moments = False
    for model, copies in ((m, most), (m, most + 3), (tiled, most + 3)):
        F, E, V = evaluate(model, copies)
        # either side keeps 2e-5 of the largest force and 1e-5 of the largest energy from the oracle
        assert np.abs(F - Fb[:1]).max() <= 2 * (2e-5 * f_scale + 2e-7)
        assert np.abs(E - Eb[:1]).max() <= 2e-5 * e_scale
        assert np.abs(V - Vb[:1]).max() <= 2e-5 * 32 * max(1.0, f_scale)
        by_moments = by_moments or not np.array_equal(F[:1], Fb[:1])
        if model is m:
            assert np.array_equal(F, np.repeat(F[:1], len(F), axis=0))      # copies agree bit for bit
    assert by_moments
    m.close()
    tiled.close()


# whole systems, by moments and (tiles of fewer rows) with every edge reading its pair's rows
@pytest.mark.parametrize("case", ["periodic", "sheared", "slab", "ghosts"])
def test_systems_by_moments_match_modes_per_edge(case):
    from paper_2608_19041_b200 import binding
    p = SMALL_PROFILES["p128_3_4"]
    blob = make_blob(p, seed=84, bias_scale=0.2, e_ref_scale=0.5)
    rng = np.random.default_rng(85)
    n, a = 14, 2.6
    pos = a * np.stack(np.meshgrid(*[np.arange(n)] * 3, indexing="ij"), -1).reshape(-1, 3) + 0.2 * rng.standard_normal((n ** 3, 3))
    cell, types = np.diag([a * n] * 3), rng.integers(0, p["T"], n ** 3).astype(np.int32)
    pbc = {"periodic": (1, 1, 1), "sheared": (1, 1, 1), "slab": (1, 1, 0), "ghosts": (0, 0, 0)}[case]
    if case == "sheared":
        shear = np.array([[1.0, 0.0, 0.0], [0.12, 1.0, 0.0], [0.07, -0.05, 1.0]])
        pos, cell = pos @ shear, cell @ shear
    dp, dt = torch.as_tensor(pos, dtype=torch.float64).cuda().contiguous(), torch.as_tensor(types).cuda()
    results = []
    for kw in dict(), dict(node_tile=MOMENT_ROWS - 1):
        m = binding.Model(blob, pair_table_mb=-1, **kw)
        if case == "ghosts":
            m.set_owned_atoms(MOMENT_ROWS + 40)
        m.build_neighbors(dp, dt, cell, pbc, 0.5)
        m.get_profile()
        out = m.compute(dp, atom_energy=True)
        assert m.get_profile()["edge_forward"][1] == 2               # edge and product; two tiles
        alone = m.compute(dp, forces=False, virial=False, atom_energy=True)
        assert torch.equal(alone["atom_energy"], out["atom_energy"]) and alone["energy"] == out["energy"]
        results.append((out["forces"].cpu().numpy(), out["atom_energy"].cpu().numpy(), out["virial"]))
        m.close()
    (F, E, V), (Fb, Eb, Vb) = results
    assert not np.array_equal(F, Fb)                                 # (they did go different ways)
    f_scale, e_scale = np.abs(Fb).max(), np.abs(Eb).max()
    assert np.abs(F - Fb).max() <= 2 * (2e-5 * f_scale + 2e-7)
    assert np.abs(E - Eb).max() <= 2e-5 * e_scale
    assert np.abs(V - Vb).max() <= 2e-5 * len(pos) * max(1.0, f_scale)
    if case == "sheared":
        Fk, near = orc.Oracle(blob).force_on(pos, types, cell, pbc, 1234)
        assert np.abs(F[1234] - Fk).max() <= 2e-5 * f_scale + 2e-7
        assert max(abs(E[k] - e) for k, e in near.items()) <= 1e-5 * e_scale


def test_a_run_by_moments_equals_evaluations_and_separate_updates():
    from paper_2608_19041_b200 import binding
    p = SMALL_PROFILES["p32_3_2"]
    blob = make_blob(p, seed=86, bias_scale=0.2)
    rng = np.random.default_rng(87)
    n, steps, dt = 13, 12, 0.001
    pos = 2.8 * np.stack(np.meshgrid(*[np.arange(n)] * 3, indexing="ij"), -1).reshape(-1, 3) + 0.1 * rng.standard_normal((n ** 3, 3))
    cell, masses = np.diag([2.8 * n] * 3), np.full(p["T"], 20.0)
    types = torch.as_tensor(rng.integers(0, p["T"], n ** 3).astype(np.int32)).cuda()
    m, ref = (binding.Model(blob, pair_table_mb=-1) for _ in range(2))
    a = torch.as_tensor(pos, dtype=torch.float64).cuda().contiguous()
    va = torch.as_tensor(rng.standard_normal(pos.shape), dtype=torch.float64).cuda().contiguous()
    b, vb = a.clone(), va.clone()
    m.build_neighbors(a, types, cell, (1, 1, 1), 1.0)
    m.set_md_state(a, va, masses)
    m.get_profile()
    e_pot, _ = m.step(steps, dt, rebuild_every=5)
    assert m.get_profile()["edge_forward"][1] == 2 * (steps + 1)
    ref.build_neighbors(b, types, cell, (1, 1, 1), 1.0)
    f = ref.compute(b)["forces"]
    inv_mass = torch.as_tensor(1.0 / masses).cuda()
    for s in range(1, steps + 1):
        binding.vv_update(b, vb, f, types, inv_mass, dt, 1, True)
        if s % 5 == 0:
            ref.build_neighbors(b, types, cell, (1, 1, 1), 1.0)
        out = ref.compute(b)
        f = out["forces"]
        binding.vv_update(b, vb, f, types, inv_mass, dt, 1, False)
    assert torch.equal(a, b) and torch.equal(va, vb) and e_pot == out["energy"]      # the same operations in the same order
    m.close()
    ref.close()
