"""First calls of a process made by several threads at once, each with a handle of its own, on every device there is."""

import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

CODE = """
import threading
import numpy as np, torch
from paper_2608_19041_b200 import binding
from workloads import SMALL_PROFILES, make_blob
p = SMALL_PROFILES["p128_3_4"]
blob = make_blob(p, seed=3, bias_scale=0.2)
rng = np.random.Generator(np.random.PCG64(1))
k = 6
sites = np.stack(np.meshgrid(*[np.arange(k)] * 3, indexing="ij"), -1).reshape(-1, 3) * 2.6
pos_h, types_h = sites + rng.uniform(-0.2, 0.2, (k ** 3, 3)), rng.integers(0, p["T"], k ** 3).astype(np.int32)
devices = torch.cuda.device_count()
paths = (2, 3, 4, 2, 3, 4, 2, 2)
jobs = []
for t, path in enumerate(paths):
    torch.cuda.set_device(t % devices)
    st = torch.cuda.Stream()
    jobs.append((t % devices, st, binding.Model(blob, mlp_path=path, stream=st), torch.tensor(pos_h, device="cuda"), torch.tensor(types_h, device="cuda")))
for d in range(devices):
    torch.cuda.synchronize(d)
gate, out = threading.Barrier(len(jobs)), [None] * len(jobs)

def work(i):
    dev, st, m, pos, types = jobs[i]
    torch.cuda.set_device(dev)
    with torch.cuda.stream(st):
        gate.wait()
        m.build_neighbors(pos, types, np.eye(3) * 2.6 * k, (1, 1, 1), 0.5)
        for _ in range(3):
            r = m.compute(pos, atom_energy=True)
        st.synchronize()
        out[i] = (r["forces"].cpu(), r["atom_energy"].cpu())

threads = [threading.Thread(target=work, args=(i,)) for i in range(len(jobs))]
[t.start() for t in threads]
[t.join() for t in threads]
ref = {path: out[i] for i, path in reversed(list(enumerate(paths)))}
for i, path in enumerate(paths):
    assert out[i] is not None, i
    assert torch.equal(out[i][0], ref[path][0]) and torch.equal(out[i][1], ref[path][1]), i
    assert torch.allclose(out[i][0], ref[2][0], rtol=0, atol=2e-5 * ref[2][0].abs().max().item())
print("same", len(jobs), devices)
"""


def test_first_calls_of_several_threads():
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    for _ in range(3):
        r = subprocess.run([sys.executable, "-c", CODE], cwd=root, capture_output=True, text=True, timeout=180)
        assert r.returncode == 0 and r.stdout.startswith("same 8"), r.stdout + r.stderr
