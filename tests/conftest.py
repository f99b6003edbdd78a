import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)


def pytest_configure(config):
    config.addinivalue_line("markers", "gpu: needs a CUDA GPU (runs the sm_103a kernels through the C-ABI)")
    config.addinivalue_line("markers", "slow: long-running check")


def _cuda_available():
    try:
        import torch
        return torch.cuda.is_available()
    except Exception:
        return False


def pytest_collection_modifyitems(config, items):
    if _cuda_available():
        return
    skip = pytest.mark.skip(reason="no CUDA device")
    for it in items:
        if "gpu" in it.keywords:
            it.add_marker(skip)


@pytest.fixture(autouse=True)
def _shapes_by_size():
    """Every test starts with launch shapes taken by size, whatever shape the test before it set."""
    yield
    rs = sys.modules.get("paper_0905_2453_gb300")
    if rs is not None and getattr(rs, "_lib", None) is not None:
        for m in (False, True):
            rs.rs_unset_launch_config(m)
