import gc
import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)


def pytest_configure(config):
    config.addinivalue_line("markers", "gpu: needs a CUDA device and the built CUDA library")


@pytest.fixture(scope="session")
def oracle_mod():
    from oracle import oracle
    oracle.lib()
    return oracle


@pytest.fixture(autouse=True)
def _collect_after_gpu_tests(request):
    """A tensor that an exception's traceback keeps lives until the collector runs; a test that
    compares the allocator's figures must not meet that moment."""
    yield
    if request.node.get_closest_marker("gpu"):
        gc.collect()
