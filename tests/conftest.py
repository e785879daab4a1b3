import gc
import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)


def pytest_configure(config):
    config.addinivalue_line("markers", "gpu: needs a GB300 (sm_103a) and the CUDA library")
    config.addinivalue_line("markers", "slow: takes more than a few seconds")


@pytest.fixture(scope="session")
def oracle_core():
    from oracle import core
    return core


@pytest.fixture(autouse=True)
def _collect_before_counting(request):
    """Tests that count the library's device buffers start without the handles that
    earlier tests left in reference cycles (an exception's frames): the collector
    would free them at a moment that depends on the number of objects alone."""
    if request.module.__name__.split(".")[-1] in ("test_gpu_failures", "test_gpu_region"):
        gc.collect()
