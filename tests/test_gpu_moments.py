"""Shared radial modes by moments of the rows (many rows, no per-pair tables) against the same kernels reading every
edge's pair rows (few rows)."""

import numpy as np
import pytest
import torch

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
    for model, copies in ((m, most), (m, most + 3), (tiled, most + 3)):
        F, E, V = evaluate(model, copies)
        # either side keeps 2e-5 of the largest force and 1e-5 of the largest energy from the oracle
        assert np.abs(F - Fb[:1]).max() <= 2 * (2e-5 * f_scale + 2e-7)
        assert np.abs(E - Eb[:1]).max() <= 2e-5 * e_scale
        assert np.abs(V - Vb[:1]).max() <= 2e-5 * 32 * max(1.0, f_scale)
        if model is m:
            assert np.array_equal(F, np.repeat(F[:1], len(F), axis=0))      # copies agree bit for bit
    m.close()
    tiled.close()
