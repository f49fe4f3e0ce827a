"""Positions as whole multiples of a quantum modulo 2^32, and the launch that ends a step of molecular dynamics."""

import numpy as np
import pytest
import torch

from oracle import dpa4c as orc
from workloads import SMALL_PROFILES, make_blob, make_system

pytestmark = pytest.mark.gpu


def _cuda(a, dtype=torch.float64):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=dtype).cuda().contiguous()


def _model(name="p16_2_0", seed=91):
    from paper_2608_19041_b200 import binding
    blob = make_blob(SMALL_PROFILES[name], seed=seed, bias_scale=0.2, e_ref_scale=0.5)
    return blob, binding.Model(blob)


@pytest.mark.parametrize("skin", [0.0, 1.999, 2.0, 2.5])     # list radii around 8, where the range of the quanta doubles
@pytest.mark.parametrize("case", ["far", "across_zero", "wide", "narrow", "sheared"])
def test_edge_vectors_from_fixed_point_positions(case, skin):
    p = SMALL_PROFILES["p16_2_0"]
    s = make_system(dict(kind="random_box", atoms=24, edges=(7.0, 8.0, 9.0), min_dist=1.6, seed=92, n_types=p["T"], masses=[1.0] * p["T"]))
    pos, types, cell, pbc = s["pos"], s["types"], np.diag(np.diag(np.asarray(s["cell"], dtype=np.float64))), (1, 1, 1)
    if case == "far":                    # a cluster far outside the range of 32 bits
        pos, cell, pbc = pos + np.array([1.0e6, -3.0e5, 777.7]), np.diag([50.0] * 3), (0, 0, 0)
    elif case == "across_zero":          # coordinates of both signs around a power of two, unfolded images
        pos = pos + np.array([-8.0, 16.0, -32.0]) + cell.diagonal() * np.array([3, -2, 5])
    elif case == "wide":                 # a box whose edge is no multiple of the range, nearly empty
        cell = np.diag([1234.567, 345.678, 77.7])
    elif case == "narrow":               # three and more images along one direction
        pos, types, cell = np.array([[0.3, 1.0, 1.0], [1.1, 4.0, 5.0], [2.0, 6.5, 7.5]]), types[:3], np.diag([2.5, 8.0, 9.0])
    elif case == "sheared":
        shear = np.array([[1.0, 0.0, 0.0], [0.3, 1.0, 0.0], [-0.2, 0.25, 1.0]])
        pos, cell = pos @ shear, cell @ shear
    blob, m = _model()
    m.build_neighbors(_cuda(pos), _cuda(types, torch.int32), cell, pbc, skin)
    out = m.compute(_cuda(pos), atom_energy=True)
    ref = orc.Oracle(blob).compute(pos, types, cell, pbc)
    # the tolerances of the parity tests: the quanta add 1.3e-9 Angstrom (rms of the rounding of two ends) to an edge
    assert np.abs(out["atom_energy"].cpu().numpy() - np.asarray(ref["E_i"])).max() <= 1e-5 * np.abs(ref["E_i"]).max()
    F = np.asarray(ref["F"])
    assert np.abs(out["forces"].cpu().numpy() - F).max() <= 2e-5 * np.abs(F).max() + 2e-7
    m.close()


# one atom, one block of rows, a ragged one, and both sides of the size up to which energies and forces are reduced in one launch
@pytest.mark.parametrize("atoms", [1, 8, 1025, 32768, 32769])
def test_steps_match_evaluations_and_separate_updates(atoms):
    from paper_2608_19041_b200 import binding
    blob, m = _model("p8_2_0", 93)
    _, ref = _model("p8_2_0", 93)
    T, dt, steps = SMALL_PROFILES["p8_2_0"]["T"], 0.001, 13         # list builds at the tenth step
    n = max(2, int(np.ceil(atoms ** (1 / 3))))
    rng = np.random.default_rng(atoms)
    pos = 3.0 * np.stack(np.meshgrid(*[np.arange(n)] * 3, indexing="ij"), -1).reshape(-1, 3)[rng.permutation(n ** 3)[:atoms]]
    pos = pos + 0.2 * rng.standard_normal(pos.shape)
    types = _cuda(rng.integers(0, T, atoms), torch.int32)
    cell, masses = np.diag([3.0 * n] * 3), np.full(T, 20.0)
    a, b = _cuda(pos), _cuda(pos)
    va, vb = _cuda(rng.standard_normal(pos.shape)), None
    vb = va.clone()
    inv_mass = _cuda(1.0 / masses)
    m.build_neighbors(a, types, cell, (1, 1, 1), 1.0)
    m.set_md_state(a, va, masses)
    e_pot, _ = m.step(steps, dt, rebuild_every=10)
    ref.build_neighbors(b, types, cell, (1, 1, 1), 1.0)
    f = ref.compute(b)["forces"]
    for s in range(1, steps + 1):
        binding.vv_update(b, vb, f, types, inv_mass, dt, 1, True)
        if s % 10 == 0:
            ref.build_neighbors(b, types, cell, (1, 1, 1), 1.0)
        out = ref.compute(b)
        f = out["forces"]
        binding.vv_update(b, vb, f, types, inv_mass, dt, 1, False)
    # the same operations in the same order
    assert torch.equal(a, b) and torch.equal(va, vb)
    assert e_pot == out["energy"]
    m.close()
    ref.close()


def test_a_stale_list_is_reported_by_the_step_that_evaluates_it():
    from paper_2608_19041_b200 import binding
    rng = np.random.default_rng(95)
    pos = 3.0 * np.stack(np.meshgrid(*[np.arange(4)] * 3, indexing="ij"), -1).reshape(-1, 3) + 0.05 * rng.standard_normal((64, 3))
    types = torch.zeros(64, dtype=torch.int32, device="cuda")
    for steps, rebuild, stale in ((3, 0, False), (6, 0, True), (10, 0, True), (12, 4, False)):
        _, m = _model("p8_2_0", 94)
        p, v = _cuda(pos), _cuda(np.tile([100.0, 0.0, 0.0], (64, 1)))     # 0.1 Angstrom a step; half the skin is 0.45
        m.build_neighbors(p, types, np.diag([12.0] * 3), (1, 1, 1), 0.9)
        m.set_md_state(p, v, np.full(SMALL_PROFILES["p8_2_0"]["T"], 1.0e9))
        if stale:
            with pytest.raises(binding.UmlmdError):
                m.step(steps, 0.001, rebuild_every=rebuild)
        else:
            m.step(steps, 0.001, rebuild_every=rebuild)
        m.close()


# list radii past those whose quanta are fine enough, and a cell of many images: edge vectors as they are at a usual list radius
@pytest.mark.parametrize("case,skin", [("open", 0.0), ("open", 9.9), ("open", 10.1), ("open", 100.0), ("open", 2500.0), ("periodic", 0.0),
                                       ("periodic", 9.9), ("periodic", 10.1), ("periodic", 100.0), ("images", 0.0), ("batch", 0.0)])
def test_edge_vectors_do_not_lose_precision_with_the_list_radius(case, skin, kernel_envelope):
    p = SMALL_PROFILES["p16_2_0"]
    s = make_system(dict(kind="random_box", atoms=24, edges=(7.0, 8.0, 9.0), min_dist=1.6, seed=92, n_types=p["T"], masses=[1.0] * p["T"]))
    pos, types, cell, pbc = s["pos"], s["types"], np.diag(np.diag(np.asarray(s["cell"], dtype=np.float64))), (0, 0, 0)
    if case == "periodic":
        cell, pbc = cell * 3.0, (1, 1, 1)
    elif case in ("images", "batch"):    # 18 images along a direction at a list radius of 6
        pos, types, cell, pbc = np.array([[0.1, 1.0, 1.0], [0.2, 5.0, 4.0]]), types[:2], np.diag([0.345, 9.0, 8.0]), (1, 1, 1)
    blob, m = _model()
    if case == "batch":
        off = np.array([0, len(pos), 2 * len(pos)])
        out = m.compute_batch(off, _cuda(np.concatenate([pos, pos])), _cuda(np.concatenate([types, types]), torch.int32), np.stack([cell, cell]), pbc,
                              atom_energy=True)
    else:
        m.build_neighbors(_cuda(pos), _cuda(types, torch.int32), cell, pbc, skin)
        out = m.compute(_cuda(pos), atom_energy=True)
    ref = orc.Oracle(blob).compute(pos, types, cell, pbc)
    E, F = np.asarray(ref["E_i"]), np.asarray(ref["F"])
    # as at a usual list radius; with quanta that grow with it atomic energies were 1.7e-6 off at the largest one
    assert np.abs(out["atom_energy"].cpu().numpy()[:len(pos)] - E).max() <= 8e-7 * np.abs(E).max()
    assert np.abs(out["forces"].cpu().numpy()[:len(pos)] - F).max() <= 8e-7 * np.abs(F).max()
    m.close()
