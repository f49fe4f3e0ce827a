"""The one-kernel MLP against the CUDA-core path where its blocks change: one atom, edges of a block, every
block size, the first size with two turns of the machine, hidden widths with one to three feature tiles, ragged
ones among them, and the sizes at which the GEMM chain takes over."""

import numpy as np
import pytest
import torch

from workloads import CONFIGS, SMALL_PROFILES, make_blob

pytestmark = pytest.mark.gpu


def _evaluate(blob, n, n_types, path):
    from paper_2608_19041_b200 import binding
    rng = np.random.Generator(np.random.PCG64(n))
    k = int(np.ceil(n ** (1 / 3)))
    sites = np.stack(np.meshgrid(*[np.arange(k)] * 3, indexing="ij"), -1).reshape(-1, 3)[:n] * 2.6
    pos = torch.tensor(sites + rng.uniform(-0.3, 0.3, (n, 3))).cuda()
    types = torch.tensor(rng.integers(0, n_types, n).astype(np.int32)).cuda()
    m = binding.Model(blob, mlp_path=path)
    m.build_neighbors(pos, types, np.eye(3) * 2.6 * k, (0, 0, 0), 0.0)
    out = m.compute(pos, atom_energy=True)
    alone = m.compute(pos, forces=False, virial=False, atom_energy=True)
    m.close()
    return out, alone


@pytest.mark.parametrize("name,sizes", [
    ("p8_2_0", (1, 16, 17, 2368, 2369, 18945)),            # F = 32
    ("p16_3_2", (33, 4737, 19000)),                        # F = 48: a ragged half tile
    ("p128_3_4", (129, 7105, 11841)),                      # F = 96, thirteen K blocks in, four column tiles out
    ("cfg2_cu4000", (2000, 14209, 18945, 37889)),          # F = 256
    ("cfg4_hea128k", (2000, 9473, 11840, 11841, 23681)),   # F = 384: one and two turns, then the chain
])
def test_matches_the_cuda_core_path(name, sizes):
    p = SMALL_PROFILES.get(name) or CONFIGS[name]["profile"]
    blob = make_blob(p, seed=50, bias_scale=0.2, e_ref_scale=0.5)
    for n in sizes:
        (ref, _), (out, alone), (tile, _) = (_evaluate(blob, n, p["T"], path) for path in (1, 2, 3))
        # As for the other tensor-core kernels: splits of 22 bits and sums of at most 544 products.  These blobs
        # are not calibrated, and where features far from O(1) cancel, every kernel of this precision is further
        # from single precision than that (F = 256: 5.3e-6): the bound is then the distance of the one-tile kernel
        # (path 3), which adds the same products in the same two accumulators per output, and half as much again.
        e_scale, f_scale = ref["atom_energy"].abs().max().item(), ref["forces"].abs().max().item()
        de = max(5e-6 * e_scale, 1.5 * (ref["atom_energy"] - tile["atom_energy"]).abs().max().item())
        df = max(1e-5 * f_scale, 1.5 * (ref["forces"] - tile["forces"]).abs().max().item()) + 1e-12
        assert (ref["atom_energy"] - out["atom_energy"]).abs().max().item() <= de, n
        assert (ref["atom_energy"] - alone["atom_energy"]).abs().max().item() <= de, n
        assert (ref["forces"] - out["forces"]).abs().max().item() <= df, n


@pytest.mark.parametrize("name,n", [("cfg2_cu4000", 14209), ("cfg4_hea128k", 11840), ("cfg4_hea128k", 8000)])
def test_one_accumulator_set_never_waits_for_a_phase_that_is_over(name, n):
    # blocks so large that tensor memory holds one set of accumulators: every pass but the first of a block then waits for
    # the epilogue before it, many times over, with a limit that an ordinary wait stays far below
    from paper_2608_19041_b200 import binding
    blob = make_blob(CONFIGS[name]["profile"], seed=51, bias_scale=0.2)
    m = binding.Model(blob, gemm_spin_limit=200000, launch_graphs=1)
    k = int(np.ceil(n ** (1 / 3)))
    sites = np.stack(np.meshgrid(*[np.arange(k)] * 3, indexing="ij"), -1).reshape(-1, 3)[:n] * 6.5      # no neighbours: the MLP is the call
    pos, types = torch.tensor(sites).cuda(), torch.zeros(n, dtype=torch.int32, device="cuda")
    m.build_neighbors(pos, types, np.eye(3) * 6.5 * k, (0, 0, 0), 0.0)
    f, e = torch.empty_like(pos), torch.empty(n, dtype=torch.float64, device="cuda")
    first = None
    for _ in range(300):
        m.compute(pos, out_forces=f, out_atom_energy=e)
        m.compute(pos, forces=False, virial=False, out_atom_energy=e)
        first = e.clone() if first is None else first
        assert torch.equal(e, first)
    m.close()
