"""List builds at the atom counts where bins and row offsets change from one block to several."""

import numpy as np
import pytest
import torch

from tests.test_gpu_scan import RC, _check_rows
from workloads import SMALL_PROFILES, make_blob

pytestmark = pytest.mark.gpu


def _model():
    from paper_2608_19041_b200 import binding
    return binding.Model(make_blob(SMALL_PROFILES["p16_2_0"], 3))      # three species


# one atom; bins in one block and in several; offsets in one block and in several
@pytest.mark.parametrize("n", [1, 31, 1023, 1024, 1025, 4095, 4096, 4097, 8192, 8193])
@pytest.mark.parametrize("case", ["periodic", "clustered", "ghosts"])
def test_rows_where_the_launches_change(n, case):
    rng = np.random.Generator(np.random.PCG64(n))
    skin = 0.5
    edge = 40.0 if case == "periodic" else 400.0
    cell, pbc = np.diag([edge, edge + 1.0, edge + 2.5]), (1, 1, 1) if case == "periodic" else (0, 1, 0)
    pos = rng.random((n, 3)) * np.diag(cell)
    if case == "clustered":                      # most bins empty, a few atoms far from the others
        pos[: n - n // 8] = pos[: n - n // 8] * 0.1 + 180.0
    if case == "ghosts":
        pos = pos * 0.08
    m = _model()
    owned = n if case != "ghosts" else n // 3
    if case == "ghosts":
        m.set_owned_atoms(owned)
    types = torch.as_tensor(rng.integers(0, 3, n), dtype=torch.int32).cuda()
    p = torch.as_tensor(pos, dtype=torch.float64).cuda().contiguous()
    m.build_neighbors(p, types, cell, pbc, skin)
    _check_rows(m, pos, cell, pbc, RC + skin, np.unique(rng.choice(n, min(n, 12))))
    out = m.compute(p, atom_energy=True)
    E = out["atom_energy"].cpu().numpy()
    assert np.all(E[owned:] == 0.0)
    if case != "ghosts" and n > 1:               # a wrong reverse slot or row sum breaks Newton's third law
        F = out["forces"].cpu().numpy()
        assert np.abs(F.sum(axis=0)).max() <= 2e-6 * max(np.abs(F).max(), 1e-6) * np.sqrt(n) * 10
    m.close()


@pytest.mark.parametrize("n", [700, 5000, 9000])
def test_bad_atoms_are_reported_at_every_size(n):
    from paper_2608_19041_b200 import binding
    rng = np.random.Generator(np.random.PCG64(n))
    cell = np.diag([40.0, 41.0, 42.0])
    pos = rng.random((n, 3)) * np.diag(cell)
    m = _model()
    good = torch.as_tensor(rng.integers(0, 3, n), dtype=torch.int32).cuda()
    p = torch.as_tensor(pos, dtype=torch.float64).cuda().contiguous()
    for value in (-1, 3):
        bad = good.clone()
        bad[n // 2] = value
        with pytest.raises(binding.UmlmdError, match="species"):
            m.build_neighbors(p, bad, cell, (1, 1, 1), 0.0)
    nan = p.clone()
    nan[n - 1, 1] = float("nan")
    with pytest.raises(binding.UmlmdError, match="finite"):
        m.build_neighbors(nan, good, cell, (1, 1, 1), 0.0)
    m.build_neighbors(p, good, cell, (1, 1, 1), 0.0)      # and nothing of it is left behind
    m.compute(p)
    off = np.array([0, n // 2, n])
    with pytest.raises(binding.UmlmdError, match="species"):
        m.compute_batch(off, p, bad, np.stack([cell, cell]), (1, 1, 1))
    assert np.isfinite(m.compute_batch(off, p, good, np.stack([cell, cell]), (1, 1, 1))["energies"]).all()
    m.close()
