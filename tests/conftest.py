import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)


def pytest_configure(config):
    config.addinivalue_line("markers", "gpu: needs a CUDA GPU (GB300, sm_103a)")
    config.addinivalue_line("markers", "slow: longer CPU test")


@pytest.fixture(autouse=True)
def shipped_pool_retention(request):
    """GPU tests run, and leave the next one to run, with the retention that
    the library's memory pool has by default (a sixteenth of the device)."""
    yield
    if request.node.get_closest_marker("gpu"):
        import torch
        from paper_2405_15197_gb300 import liblm
        if torch.cuda.is_available():
            liblm.lm_pool_retain(torch.cuda.mem_get_info()[1] // 16)
