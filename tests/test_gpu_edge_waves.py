"""Edge kernels at the row counts that one wave of 32 warps per SM holds and 24 do not (3553 to 4736): the backward kernel
there has a variant of fewer registers, compared with the wider one on the same frames in a larger call."""

import numpy as np
import pytest
import torch

from workloads import SMALL_PROFILES, make_blob, make_system

pytestmark = pytest.mark.gpu

WARPS_24, WARPS_32 = 148 * 24, 148 * 32


@pytest.mark.parametrize("pair_table_mb", [-1, 0], ids=["pair_cache", "pair_tables"])
@pytest.mark.parametrize("name", sorted(n for n, p in SMALL_PROFILES.items() if p["C0"] <= 64))
def test_one_wave_of_more_warps_matches_two_of_fewer(name, pair_table_mb):
    from paper_2608_19041_b200 import binding
    p = SMALL_PROFILES[name]
    s = make_system(dict(kind="random_box", atoms=37, edges=(8.5, 9.0, 9.5), min_dist=1.6, seed=91, n_types=p["T"], masses=[1.0] * p["T"]))
    cell = np.diag(np.diag(np.asarray(s["cell"], dtype=np.float64)))
    m = binding.Model(make_blob(p, seed=93, bias_scale=0.2, e_ref_scale=0.5), pair_table_mb=pair_table_mb)

    def evaluate(copies):
        out = m.compute_batch(np.arange(copies + 1) * 37, torch.as_tensor(np.tile(s["pos"], (copies, 1)), dtype=torch.float64).cuda().contiguous(),
                              torch.as_tensor(np.tile(s["types"], copies), dtype=torch.int32).cuda().contiguous(), np.stack([cell] * copies),
                              (1, 1, 1), atom_energy=True)
        return (out["forces"].cpu().numpy().reshape(copies, 37, 3), out["atom_energy"].cpu().numpy().reshape(copies, 37),
                np.asarray(out["virials"]).reshape(copies, -1))

    wide = evaluate(WARPS_32 // 37 + 1)                       # 4773 rows: 24 warps per SM, in two waves
    f_scale, e_scale = np.abs(wide[0]).max(), np.abs(wide[1]).max()
    for copies in (WARPS_24 // 37 + 1, WARPS_32 // 37):       # 3589 and 4736 rows
        assert WARPS_24 < 37 * copies <= WARPS_32
        F, E, V = evaluate(copies)
        # either side keeps 2e-5 of the largest force and 1e-5 of the largest energy from the oracle
        assert np.abs(F - wide[0][:copies]).max() <= 2 * (2e-5 * f_scale + 2e-7)
        assert np.abs(E - wide[1][:copies]).max() <= 2e-5 * e_scale
        assert np.abs(V - wide[2][:copies]).max() <= 2e-5 * 37 * max(1.0, f_scale)
        assert np.array_equal(F, np.repeat(F[:1], copies, axis=0))
    m.close()
