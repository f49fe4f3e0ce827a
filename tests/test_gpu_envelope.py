"""The envelope of the edge kernels against its definition: no error that all edges share."""

import numpy as np
import pytest
import torch

from oracle import dpa4c as orc
from workloads import SMALL_PROFILES, make_blob

pytestmark = pytest.mark.gpu


# cutoffs that are and are not single-precision numbers; widths whose kernels form 1 / rc in either way
@pytest.mark.parametrize("name", ["p16_2_0", "p128_2_0"])
@pytest.mark.parametrize("rc", [5.2, 6.0, 7.0])
def test_envelope_sums_have_no_common_error(rc, name):
    from paper_2608_19041_b200 import binding
    p = dict(SMALL_PROFILES[name], rc=rc)
    blob = make_blob(p, seed=61)
    o, m = orc.Oracle(blob), binding.Model(blob)
    rng = np.random.default_rng(62)
    pos = 2.3 * np.stack(np.meshgrid(*[np.arange(11)] * 3, indexing="ij"), -1).reshape(-1, 3) + 0.2 * rng.standard_normal((1331, 3))
    cell, types = np.diag([2.3 * 11] * 3), np.zeros(1331, dtype=np.int32)
    gpu = torch.as_tensor(pos, dtype=torch.float64).cuda().contiguous()
    m.build_neighbors(gpu, torch.as_tensor(types).cuda(), cell, (1, 1, 1), 0.0)
    m.compute(gpu, forces=False, virial=False)
    s0, s1 = m.get_intermediates()[0][:, -2:].cpu().numpy().astype(np.float64).T
    m.close()
    w = orc.wrap_positions(pos, cell, (1, 1, 1))
    dst, _, rij = orc.rows_to_edges(orc.neighbor_rows(w, cell, (1, 1, 1), rc), np.arange(1331), w, cell)
    chi = orc.envelope(torch.from_numpy(np.sqrt((rij ** 2).sum(axis=1) + orc.EPS_REG ** 2)), rc).numpy()
    # the powers' relative errors: chi is good to 2^-24 and a few roundings each way, which average out over 1331 rows of 40 to
    # 100 edges: 2^-24 times four over the root of 50,000 is 1.1e-9
    for got, power in ((s0, 2), (s1, 4)):
        ref = np.zeros(1331)
        np.add.at(ref, dst, chi ** power)
        assert abs(got.sum() / ref.sum() - 1) <= 1e-8 * power, (power, got.sum() / ref.sum() - 1)
        assert np.sqrt(((got - ref) ** 2).mean()) <= 2.0 ** -24 * power * ref.mean()
