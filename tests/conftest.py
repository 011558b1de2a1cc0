import os
import sys
from pathlib import Path

import pytest

ROOT = Path(__file__).resolve().parent.parent
if str(ROOT) not in sys.path:
    sys.path.insert(0, str(ROOT))


def pytest_configure(config):
    config.addinivalue_line("markers", "gpu: needs a CUDA device (runs the hand-written kernels through the C ABI)")


def pytest_collection_modifyitems(config, items):
    # A GPU test on a machine without one is a skip, never a silent CPU fallback.
    try:
        import torch
        has_gpu = torch.cuda.is_available()
    except Exception:
        has_gpu = False
    if not has_gpu:
        skip = pytest.mark.skip(reason="no CUDA device")
        for it in items:
            if "gpu" in it.keywords:
                it.add_marker(skip)


@pytest.fixture(autouse=True)
def _collect_after_gpu_test(request):
    """A test that catches an error keeps its frame, and with it a context's device buffers, alive in a reference cycle.
    They go with the test, not whenever the collector next runs -- which may be between two readings of the allocator in
    a later one."""
    yield
    if "gpu" in request.node.keywords:
        import gc
        gc.collect()
