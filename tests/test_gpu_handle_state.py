"""What a handle keeps from call to call: flags across replayed sequences, buffers across systems of growing size."""

import numpy as np
import pytest
import torch

from workloads import CONFIGS, SMALL_PROFILES, make_blob

pytestmark = pytest.mark.gpu


def _box(n, n_types, seed=0, a=2.6):
    rng = np.random.Generator(np.random.PCG64(seed))
    k = int(np.ceil(n ** (1 / 3)))
    sites = np.stack(np.meshgrid(*[np.arange(k)] * 3, indexing="ij"), -1).reshape(-1, 3)[:n] * a
    pos = torch.tensor(sites + rng.uniform(-0.2, 0.2, (n, 3))).cuda()
    types = torch.tensor(rng.integers(0, n_types, n).astype(np.int32)).cuda()
    return pos, types, np.eye(3) * a * k


@pytest.mark.parametrize("driver", ["nve", "nvt"])
def test_replayed_evaluations_keep_track_of_what_the_buffers_hold(driver):
    from paper_2608_19041_b200 import binding
    p = SMALL_PROFILES["p16_2_0"]
    blob = make_blob(p, seed=3, bias_scale=0.2)
    start, types, cell = _box(150, p["T"], seed=4)
    results = []
    for graphs in (-1, 1):
        m = binding.Model(blob, launch_graphs=graphs)
        pos, vel = start.clone(), torch.zeros_like(start)
        ea, f = torch.empty(150, dtype=torch.float64, device="cuda"), torch.empty_like(pos)
        m.build_neighbors(pos, types, cell, (1, 1, 1), 1.0)
        m.set_md_state(pos, vel, [20.0] * p["T"])

        def energy():
            m.compute(pos, forces=False, virial=False, out_atom_energy=ea)

        def steps(n):
            return m.step(n, 1e-4) if driver == "nve" else m.step_nvt(n, 1e-4, 300.0, 0.1)

        for _ in range(3):                # plain, recorded, replayed
            energy()
        steps(1)                          # its only step runs plain and leaves gradients
        energy()                          # replayed: forward values again
        state, desc = m.get_intermediates()
        with pytest.raises(binding.UmlmdError) as e:
            m.atom_virial()
        assert e.value.code == -1
        # the other way round: the last evaluation with forces is a replayed one
        steps(4)
        energy()
        out = [m.compute(pos, out_forces=f) for _ in range(3)][-1]
        w = m.atom_virial()
        assert np.abs(w.sum(dim=0).cpu().numpy() - out["virial"]).max() <= 1e-6 * w.abs().sum().item()
        results.append((state.clone(), desc.clone(), w.clone(), out["energy"]))
        assert (m.query()["graph_replays"] > 0) == (graphs == 1)
        m.close()
    for a, b in zip(*results):
        assert torch.equal(a, b) if isinstance(a, torch.Tensor) else a == b


def test_md_state_of_a_larger_system_gets_a_larger_force_buffer():
    # accounting alone: nothing is launched on the buffer
    from paper_2608_19041_b200 import binding
    p = SMALL_PROFILES["p16_2_0"]
    m = binding.Model(make_blob(p, seed=3))
    for n, grown in ((300, None), (880, 24 * (880 - 300)), (881, 0), (400, 0)):      # (buffers are padded by 16 elements)
        pos, types, cell = _box(n, p["T"])
        m.build_neighbors(pos, types, cell, (1, 1, 1), 1.0)
        held = m.query()["device_bytes"]
        m.set_md_state(pos, torch.zeros_like(pos), [20.0] * p["T"])
        assert grown is None or m.query()["device_bytes"] - held == grown, n
    m.close()


def test_md_after_a_smaller_system_on_the_same_handle():
    from paper_2608_19041_b200 import binding
    p = SMALL_PROFILES["p16_2_0"]
    blob = make_blob(p, seed=3, bias_scale=0.2)
    used, results = binding.Model(blob), []
    for n, m in ((300, used), (880, used), (880, binding.Model(blob))):
        pos, types, cell = _box(n, p["T"], seed=5)
        vel = torch.zeros_like(pos)
        m.build_neighbors(pos, types, cell, (1, 1, 1), 1.0)
        m.set_md_state(pos, vel, [20.0] * p["T"])
        e = m.step(12, 1e-4, rebuild_every=5)
        results.append((e, pos, vel))
    (ea, pa, va), (eb, pb, vb) = results[1:]
    assert ea == eb and torch.equal(pa, pb) and torch.equal(va, vb)


def test_a_failed_allocation_leaves_no_list_and_is_made_up_for():
    """Builds of a large system with less and less device memory to spare fail wherever the memory runs out; after each
    the handle refuses to evaluate, and evaluates a small system as before."""
    from paper_2608_19041_b200 import binding
    p = SMALL_PROFILES["p128_2_0"]
    small, big = _box(600, p["T"], seed=6), _box(60000, p["T"], seed=7)
    blob = make_blob(p, seed=3, bias_scale=0.2)

    def evaluate(m):
        m.build_neighbors(*small, (1, 1, 1), 1.0)
        out = m.compute(small[0], atom_energy=True)
        return out["forces"], out["atom_energy"]

    m = binding.Model(blob)
    ref = evaluate(m)
    m.close()
    failed = 0
    for spare_mb in (24, 64, 100, 140, 180, 240, 300, 380, 460, 560, 700):
        m = binding.Model(blob)
        if spare_mb % 100:                               # on a handle in use, and on one whose first build it is
            evaluate(m)
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        hog = torch.empty(max(torch.cuda.mem_get_info()[0] - (spare_mb << 20), 1), dtype=torch.uint8, device="cuda")
        try:
            m.build_neighbors(*big, (1, 1, 1), 1.0)
        except binding.UmlmdError as e:
            assert e.code == -8
            failed += 1
            lib = binding.lib()
            assert lib.umlmd_compute(m._h, big[0].data_ptr(), None, None, None, None) == -5
            assert lib.umlmd_step(m._h, 1, 0.001, 0, None, None) == -5
            assert lib.umlmd_atom_virial(m._h, big[0].data_ptr()) == -5
        del hog
        torch.cuda.empty_cache()
        for a, b in zip(evaluate(m), ref):
            assert torch.equal(a, b), spare_mb
        m.close()
    assert failed >= 6


def _held(blob, box, **kw):
    """Device memory that a handle takes for its first build."""
    from paper_2608_19041_b200 import binding
    m = binding.Model(blob, **kw)
    before = m.query()["device_bytes"]
    m.build_neighbors(*box, (0, 0, 0), 0.0)
    held = m.query()["device_bytes"] - before
    m.close()
    return held


def test_the_first_build_allocates_what_the_system_uses():
    # the one-kernel MLP's areas only where the rule takes it: 24,000 atoms at F = 384 go through the chain of GEMMs
    p = CONFIGS["cfg4_hea128k"]["profile"]
    blob = make_blob(p, seed=3)
    box = _box(24000, p["T"], a=6.5)
    assert _held(blob, box) == _held(blob, box, mlp_path=3)
    # the cubic pieces where per-pair tables are made from them, the value and product tables where they are read themselves
    p = SMALL_PROFILES["p128_2_0"]
    blob = make_blob(p, seed=3)
    box = _box(64, p["T"])
    rows, pad = 3000, 16
    cubic, quadratic = 12 * rows * 128 + pad, 8 * rows * 128 + pad
    tables = 4 * (32 + p["T"] ** 2 * 2 * rows * 2 * 128 + pad)
    assert _held(blob, box) - _held(blob, box, pair_table_mb=-1) == tables + cubic - 2 * quadratic


def test_a_limit_on_pair_tables_bounds_their_memory():
    # three species at C0 = 128: nine pairs of 5.9 MiB, 52.8 in all (39.6 if only the cubic pieces are counted)
    p = SMALL_PROFILES["p128_2_0"]
    blob = make_blob(p, seed=3)
    box = _box(64, p["T"])
    without = _held(blob, box, pair_table_mb=-1)
    for limit, built in ((1, False), (45, False), (52, False), (53, True), (400, True), (0, True)):
        held = _held(blob, box, pair_table_mb=limit) - without
        assert (held > 0) == built, limit
        assert held <= (limit or 320) << 20, limit
