import gc
import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)


def pytest_configure(config):
    config.addinivalue_line("markers", "gpu: needs a CUDA device (B200) and the built native library")


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


@pytest.fixture(scope="session", autouse=True)
def native_library():
    """Builds libbsr.so in-tree when it is missing and nvcc is present (cross-compiles without a GPU)."""
    from paper_2405_10951_b200 import binding, build
    if not os.path.exists(binding.LIB_PATH):
        build.build()
    yield


@pytest.fixture(scope="module", autouse=True)
def earlier_modules_collected():
    """Device tensors in reference cycles (a caught exception's frames) go now, not in the middle of a test that watches the allocator."""
    gc.collect()
    yield
