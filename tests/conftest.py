import gc
import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)


def pytest_configure(config):
    config.addinivalue_line("markers", "gpu: needs a CUDA GPU (sm_103a) and the built libpin.so")
    config.addinivalue_line("markers", "slow: long-running CPU test")


@pytest.fixture(scope="session")
def gpu_available():
    import torch
    return torch.cuda.is_available()


@pytest.fixture(autouse=True)
def _collect_before(request):
    """A plan of an earlier test that sits in a reference cycle (the traceback
    that pytest.raises keeps) is freed here, not in the middle of a test that
    compares the device's free memory before and after."""
    if request.node.get_closest_marker("gpu"):
        gc.collect()
