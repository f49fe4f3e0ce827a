import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)


def pytest_configure(config):
    config.addinivalue_line("markers", "gpu: test needs a CUDA device (B200)")


def pytest_collection_modifyitems(config, items):
    try:
        import torch
        has_gpu = torch.cuda.is_available()
    except Exception:
        has_gpu = False
    if has_gpu:
        return
    skip = pytest.mark.skip(reason="no CUDA device")
    for item in items:
        if "gpu" in item.keywords:
            item.add_marker(skip)


@pytest.fixture
def kernel_envelope(monkeypatch):
    """The oracle's envelope with the cutoff that the edge kernels' single-precision 1 / rc stands for: what that factor is off, all
    edges share (1e-7 of chi at rc = 6), and a test of something smaller has to leave it out."""
    import numpy as np

    from oracle import dpa4c as orc
    exact = orc.envelope
    monkeypatch.setattr(orc, "envelope", lambda rho, rc: exact(rho, 1.0 / float(np.float32(1.0) / np.float32(rc))))
