import gc
import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)


def pytest_configure(config):
    config.addinivalue_line("markers", "gpu: needs a CUDA GPU (GB300, sm_103a)")
    config.addinivalue_line("markers", "slow: oracle runs that take tens of seconds")


@pytest.fixture(autouse=True, scope="module")
def _collect_contexts():
    """A module's contexts give their device memory back before the next one
    starts (a test there may compare the free memory before and after)."""
    yield
    gc.collect()
