"""Scalar channels by splines (one species, many rows) against the same kernels reading the pair's tables (few rows)."""

import os
import subprocess
import sys

import numpy as np
import pytest
import torch

from oracle import dpa4c as orc
from tests.test_host_tables import _steep_blob
from workloads import SMALL_PROFILES, make_blob, make_system

pytestmark = pytest.mark.gpu

SPLINE_ROWS = 8192      # the fewest rows that take the way over splines


def _frames():
    # 29 atoms with long rows, some closer than any material has them, and three with rows of at most two edges
    dense = make_system(dict(kind="random_box", atoms=29, edges=(4.6, 5.0, 5.4), min_dist=0.9, seed=81, n_types=1, masses=[1.0]))
    sparse = make_system(dict(kind="random_box", atoms=3, edges=(30.0, 30.0, 30.0), min_dist=1.6, seed=82, n_types=1, masses=[1.0]))
    sparse["pos"][:2] = [[3.0, 3.0, 3.0], [4.7, 3.2, 3.1]]
    return (29, 3), [np.diag(np.diag(np.asarray(f["cell"], dtype=np.float64))) for f in (dense, sparse)], np.concatenate([dense["pos"], sparse["pos"]])


def _evaluate(model, copies, species=0):
    sizes, cells, frame = _frames()
    off = np.concatenate([[0], np.cumsum(np.tile(sizes, copies))])
    pos = torch.as_tensor(np.tile(frame, (copies, 1)), dtype=torch.float64).cuda().contiguous()
    types = torch.full((32 * copies,), species, dtype=torch.int32, device="cuda")
    out = model.compute_batch(off, pos, types, np.stack(cells * copies), (1, 1, 1), atom_energy=True)
    return (out["forces"].cpu().numpy().reshape(copies, 32, 3), out["atom_energy"].cpu().numpy().reshape(copies, 32),
            np.asarray(out["virials"]).reshape(copies, 2, -1))


def _compare(a, b):
    (F, E, V), (Fb, Eb, Vb) = a, b
    f_scale, e_scale = np.abs(Fb).max(), np.abs(Eb).max()
    # either side keeps 2e-5 of the largest force and 1e-5 of the largest energy from the oracle
    assert np.abs(F - Fb[:1]).max() <= 2 * (2e-5 * f_scale + 2e-7)
    assert np.abs(E - Eb[:1]).max() <= 2e-5 * e_scale
    assert np.abs(V - Vb[:1]).max() <= 2e-5 * 32 * max(1.0, f_scale)


@pytest.mark.parametrize("basis", ["bessel", "gaussian"])
@pytest.mark.parametrize("name", ["p64_3_8", "p128_2_0", "p128_3_4", "p128_4_4"])
def test_splines_match_tables(name, basis):
    from paper_2608_19041_b200 import binding
    p = SMALL_PROFILES[name]
    blob = make_blob(p, seed=83, bias_scale=0.2, e_ref_scale=0.5, basis=basis)
    m = binding.Model(blob)
    tiled = binding.Model(blob, node_tile=SPLINE_ROWS + 1)       # a tile by splines, one of 95 rows without
    most = SPLINE_ROWS // 32
    ref = _evaluate(m, most - 1)                                  # tables
    by_splines = False
    for model, copies in ((m, most), (m, most + 3), (tiled, most + 3)):
        out = _evaluate(model, copies)
        _compare(out, ref)
        by_splines = by_splines or not np.array_equal(out[0][:1], ref[0][:1])
        if model is m:
            assert np.array_equal(out[0], np.repeat(out[0][:1], copies, axis=0))      # copies agree bit for bit
    assert by_splines
    _compare(_evaluate(m, most, species=p["T"] - 1), _evaluate(m, most - 1, species=p["T"] - 1))     # another pair, same fit
    m.close()
    tiled.close()


@pytest.mark.parametrize("case", ["steep", "coarse"])
def test_maps_without_a_fit_keep_their_tables(case):
    from paper_2608_19041_b200 import binding
    p = SMALL_PROFILES["p128_3_4"]
    # a high frequency that a few hundred intervals cannot follow; a table with fewer knots than intervals
    m = binding.Model(_steep_blob(p, 3, 1.0, 250)) if case == "steep" else binding.Model(make_blob(p, seed=83), table_dx=0.05)
    most = SPLINE_ROWS // 32
    a, b = _evaluate(m, most), _evaluate(m, most - 1)
    assert np.array_equal(a[0][:-1], b[0]) and np.array_equal(a[1][:-1], b[1])
    m.close()


def _lattice(atoms, spacing, jitter, seed):
    n = int(np.ceil(atoms ** (1 / 3) - 1e-9))
    rng = np.random.default_rng(seed)
    pos = spacing * np.stack(np.meshgrid(*[np.arange(n)] * 3, indexing="ij"), -1).reshape(-1, 3)[rng.permutation(n ** 3)[:atoms]]
    return pos + jitter * rng.standard_normal(pos.shape), np.diag([spacing * n] * 3)


def _row_sums(blob, m, pos, cell, species, centers):
    """Scalar channels' sums of the given rows: the library's, and those of the oracle."""
    types = np.full(len(pos), species, dtype=np.int32)
    p = torch.as_tensor(pos, dtype=torch.float64).cuda().contiguous()
    m.build_neighbors(p, torch.as_tensor(types).cuda(), cell, (1, 1, 1), 0.0)
    m.compute(p, forces=False, virial=False)
    C0 = m.query()["C0"]
    got = m.get_intermediates()[0][:, :C0].cpu().numpy()[centers].astype(np.float64)
    o = orc.Oracle(blob)
    w = orc.wrap_positions(pos, cell, (1, 1, 1))
    dst, _, rij = orc.rows_to_edges(orc.neighbor_rows(w, cell, (1, 1, 1), o.p["rc"], centers=centers), centers, w, cell)
    t = torch.full((len(dst),), species, dtype=torch.int64)
    A = orc.aggregate(o.p, o.prm, o.pair, len(centers), torch.from_numpy(dst), t, t, torch.from_numpy(rij))[0]
    return got, A[0].reshape(len(centers), C0).numpy()


# neighbours at few distances: the weights of successive edges fall on the same or on the next places of the row; odd counts
@pytest.mark.parametrize("jitter", [0.004, 0.1])
@pytest.mark.parametrize("name,spacing", [("p64_3_8", 1.6), ("p128_2_0", 1.9)])
def test_row_sums_follow_the_definition(name, spacing, jitter, kernel_envelope):
    from paper_2608_19041_b200 import binding
    blob = make_blob(SMALL_PROFILES[name], seed=84, bias_scale=0.2, e_ref_scale=0.5)
    m = binding.Model(blob)
    pos, cell = _lattice(SPLINE_ROWS + 7, spacing, jitter, 85)
    got, ref = _row_sums(blob, m, pos, cell, 0, np.arange(5, len(pos), 8))
    m.close()
    # a row's sum of products has the rounding of its 168 single-precision terms in two levels: below 2^-22 of the sums' rms,
    # six times that for the largest of 65,000 and more; a weight that is lost is 1e-3 and more
    rms = np.sqrt((ref ** 2).mean())
    err = got - ref
    assert np.sqrt((err ** 2).mean()) <= 2.0 ** -22 * rms
    assert np.abs(err).max() <= 6 * 2.0 ** -22 * rms


# whole systems, by splines and (tiles of fewer rows) by tables
@pytest.mark.parametrize("case", ["periodic", "sheared", "slab", "ghosts"])
@pytest.mark.parametrize("name,spacing", [("p64_3_8", 1.6), ("p128_2_0", 1.9)])
def test_systems_by_splines_match_tables(name, spacing, case):
    from paper_2608_19041_b200 import binding
    blob = make_blob(SMALL_PROFILES[name], seed=88, bias_scale=0.2, e_ref_scale=0.5)
    pos, cell = _lattice(21 ** 3, spacing, 0.1, 89)
    pbc = {"periodic": (1, 1, 1), "sheared": (1, 1, 1), "slab": (1, 1, 0), "ghosts": (0, 0, 0)}[case]
    if case == "sheared":
        shear = np.array([[1.0, 0.0, 0.0], [0.12, 1.0, 0.0], [0.07, -0.05, 1.0]])
        pos, cell = pos @ shear, cell @ shear
    types = torch.ones(len(pos), dtype=torch.int32, device="cuda")
    p = torch.as_tensor(pos, dtype=torch.float64).cuda().contiguous()
    results = []
    for kw, launches in (dict(), 2), (dict(node_tile=SPLINE_ROWS - 1), 2):            # edge and product; two tiles
        m = binding.Model(blob, **kw)
        if case == "ghosts":
            m.set_owned_atoms(SPLINE_ROWS + 40)
        m.build_neighbors(p, types, cell, pbc, 0.5)
        m.get_profile()
        out = m.compute(p, atom_energy=True)
        assert m.get_profile()["edge_forward"][1] == launches
        alone = m.compute(p, forces=False, virial=False, atom_energy=True)
        assert torch.equal(alone["atom_energy"], out["atom_energy"]) and alone["energy"] == out["energy"]
        results.append((out["forces"].cpu().numpy(), out["atom_energy"].cpu().numpy(), out["virial"]))
        m.close()
    (F, E, V), (Fb, Eb, Vb) = results
    assert not np.array_equal(F, Fb)                   # (they did go different ways)
    # either side keeps 2e-5 of the largest force and 1e-5 of the largest energy from the oracle
    f_scale, e_scale = np.abs(Fb).max(), np.abs(Eb).max()
    assert np.abs(F - Fb).max() <= 2 * (2e-5 * f_scale + 2e-7)
    assert np.abs(E - Eb).max() <= 2e-5 * e_scale
    assert np.abs(V - Vb).max() <= 2e-5 * len(pos) * max(1.0, f_scale)
    if case == "sheared":
        Fk, near = orc.Oracle(blob).force_on(pos, np.ones(len(pos), dtype=np.int32), cell, pbc, 4567)
        assert np.abs(F[4567] - Fk).max() <= 2e-5 * f_scale + 2e-7
        assert max(abs(E[a] - e) for a, e in near.items()) <= 1e-5 * e_scale


def test_a_run_by_splines_follows_the_run_by_tables():
    from paper_2608_19041_b200 import binding
    blob = make_blob(SMALL_PROFILES["p128_2_0"], seed=88, bias_scale=0.2)
    pos, cell = _lattice(21 ** 3, 1.9, 0.05, 90)
    vel = np.random.default_rng(91).standard_normal(pos.shape)
    masses = np.full(SMALL_PROFILES["p128_2_0"]["T"], 20.0)
    runs = []
    for kw in dict(), dict(node_tile=SPLINE_ROWS - 1):
        m = binding.Model(blob, **kw)
        p, v = (torch.as_tensor(x, dtype=torch.float64).cuda().contiguous() for x in (pos, vel))
        m.build_neighbors(p, torch.zeros(len(pos), dtype=torch.int32, device="cuda"), cell, (1, 1, 1), 0.6)
        m.set_md_state(p, v, masses)
        e = m.step(13, 0.0005, rebuild_every=5)
        f = m.compute(p)["forces"]
        runs.append((p, v, f, sum(e)))
        m.close()
    (p, v, f, e), (pb, vb, fb, eb) = runs
    # forces agree to 4e-5 of the largest; the positions' difference after n steps is at most n^2 / 2 times what one step makes of that
    f_scale = fb.abs().max().item()
    step = 4e-5 * f_scale / 20.0 * 9648.53321 * 0.0005 ** 2
    assert (p - pb).abs().max().item() <= 13 ** 2 / 2 * step
    assert (f - fb).abs().max().item() <= 8e-5 * f_scale
    assert abs(e - eb) <= 2e-5 * len(pos)


# some 97 and 79 listed neighbours on average: either side of where splines are taken at this width
@pytest.mark.parametrize("spacing,growth", [(2.29, 0.02), (2.33, -0.02)])
def test_a_run_keeps_the_way_its_list_was_built_for(spacing, growth):
    from paper_2608_19041_b200 import binding
    m = binding.Model(make_blob(SMALL_PROFILES["p128_2_0"], seed=84))
    pos, cell = _lattice(21 ** 3, spacing, 0.02, 86)
    steps, dt = 10, 0.001
    pos = pos - pos.mean(axis=0)
    vel = pos * (growth / (steps * dt))                # the cluster grows or shrinks by 2 % in all
    p, v = (torch.as_tensor(x, dtype=torch.float64).cuda().contiguous() for x in (pos, vel))
    types = torch.zeros(len(pos), dtype=torch.int32, device="cuda")
    m.build_neighbors(p, types, 4 * cell, (0, 0, 0), 0.9)
    listed = [m.query()["n_edges"] / len(pos)]
    m.get_profile()
    m.compute(p)
    per_call = m.get_profile()["edge_forward"][1]      # one launch more by splines
    assert per_call == (2 if growth > 0 else 1)
    m.set_md_state(p, v, np.full(SMALL_PROFILES["p128_2_0"]["T"], 1.0e9))
    m.step(steps, dt, rebuild_every=2)
    listed.append(m.query()["n_edges"] / len(pos))
    assert min(listed) < 90 < max(listed)              # (the mean row has crossed the switch)
    assert m.get_profile()["edge_forward"][1] == (steps + 1) * per_call
    m.close()


THREADS = """
import threading
import numpy as np, torch
from paper_2608_19041_b200 import binding
from workloads import SMALL_PROFILES, make_blob
import tests.test_gpu_splines as base
# (models whose kernels are the same and whose rows of spline weights are not)
blobs = [make_blob(SMALL_PROFILES["p64_3_8"], seed=83, bias_scale=0.2, e_ref_scale=0.5, basis=b) for b in ("bessel", "gaussian")]
pos, cell = base._lattice(8200, 1.6, 0.05, 87)
jobs = []
for t in range(4):
    st = torch.cuda.Stream()
    jobs.append((st, binding.Model(blobs[t % 2], stream=st, launch_graphs=-1), torch.tensor(pos, device="cuda"), torch.zeros(len(pos), dtype=torch.int32, device="cuda")))
torch.cuda.synchronize()
gate, out = threading.Barrier(len(jobs)), [None] * len(jobs)

def work(i):
    st, m, p, types = jobs[i]
    with torch.cuda.stream(st):
        m.build_neighbors(p, types, cell, (1, 1, 1), 0.0)
        ref = m.compute(p)["forces"].clone()
        gate.wait()
        same = True
        for _ in range(300):
            same = same and torch.equal(m.compute(p)["forces"], ref)
        out[i] = same

threads = [threading.Thread(target=work, args=(i,)) for i in range(len(jobs))]
[t.start() for t in threads]
[t.join() for t in threads]
print(out)
"""


def test_models_with_other_rows_of_weights_in_several_threads():
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", THREADS], cwd=root, capture_output=True, text=True, timeout=180)
    assert r.returncode == 0 and r.stdout.strip() == str([True] * 4), r.stdout + r.stderr
