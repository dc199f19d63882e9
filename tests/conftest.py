import gc
import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)


def pytest_configure(config):
    config.addinivalue_line("markers", "gpu: needs a CUDA GPU (GB300, sm_103a)")


@pytest.fixture(autouse=True)
def _collect_garbage(request):
    """Tensors that a GPU test leaves in reference cycles are freed after it,
    not while a later test compares the allocator's byte counts."""
    yield
    if request.node.get_closest_marker("gpu"):
        gc.collect()
