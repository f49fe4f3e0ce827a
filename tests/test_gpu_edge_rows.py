"""Edge kernels with the warps of a block on one row (few rows) against the same kernels with a warp per row."""

import numpy as np
import pytest
import torch

from workloads import SMALL_PROFILES, make_blob, make_system

pytestmark = pytest.mark.gpu

SPLIT_ROWS = 1184       # the most rows that are shared among the warps of a block


@pytest.mark.parametrize("pair_table_mb", [-1, 0], ids=["pair_cache", "pair_tables"])
@pytest.mark.parametrize("name", sorted(SMALL_PROFILES))
def test_shared_rows_match_a_warp_per_row(name, pair_table_mb):
    from paper_2608_19041_b200 import binding
    p = SMALL_PROFILES[name]
    masses = [1.0] * p["T"]
    # 29 atoms with full rows (several batches per quarter), three with rows of at most two edges (empty quarters)
    dense = make_system(dict(kind="random_box", atoms=29, edges=(8.0, 8.5, 9.0), min_dist=1.6, seed=81, n_types=p["T"], masses=masses))
    sparse = make_system(dict(kind="random_box", atoms=3, edges=(30.0, 30.0, 30.0), min_dist=1.6, seed=82, n_types=p["T"], masses=masses))
    sparse["pos"][:2] = [[3.0, 3.0, 3.0], [4.7, 3.2, 3.1]]
    sizes, cells = (29, 3), [np.diag(np.diag(np.asarray(f["cell"], dtype=np.float64))) for f in (dense, sparse)]
    m = binding.Model(make_blob(p, seed=83, bias_scale=0.2, e_ref_scale=0.5), pair_table_mb=pair_table_mb)

    def evaluate(copies):
        off = np.concatenate([[0], np.cumsum(np.tile(sizes, copies))])
        pos = np.tile(np.concatenate([dense["pos"], sparse["pos"]]), (copies, 1))
        types = np.tile(np.concatenate([dense["types"], sparse["types"]]), copies)
        out = m.compute_batch(off, torch.as_tensor(pos, dtype=torch.float64).cuda().contiguous(),
                              torch.as_tensor(types, dtype=torch.int32).cuda().contiguous(),
                              np.stack(cells * copies), (1, 1, 1), atom_energy=True)
        return (out["forces"].cpu().numpy().reshape(copies, 32, 3), out["atom_energy"].cpu().numpy().reshape(copies, 32),
                np.asarray(out["virials"]).reshape(copies, 2, -1))

    most = SPLIT_ROWS // 32
    Fa, Ea, Va = evaluate(most)              # the largest shared call
    Fb, Eb, Vb = evaluate(most + 1)          # a warp per row
    Fc, Ec, Vc = evaluate(1)                 # the smallest
    # either side keeps 2e-5 of the largest force and 1e-5 of the largest energy from the oracle
    f_scale, e_scale = np.abs(Fb).max(), np.abs(Eb).max()
    for F, E, V in ((Fa, Ea, Va), (Fc, Ec, Vc)):
        assert np.abs(F - Fb[:len(F)]).max() <= 2 * (2e-5 * f_scale + 2e-7)
        assert np.abs(E - Eb[:len(E)]).max() <= 2e-5 * e_scale
        assert np.abs(V - Vb[:len(V)]).max() <= 2e-5 * 32 * max(1.0, f_scale)
        assert np.array_equal(F, np.repeat(F[:1], len(F), axis=0))      # copies agree bit for bit
    m.close()
