import gc
import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)


def pytest_configure(config):
    config.addinivalue_line("markers", "gpu: needs a CUDA GPU (GB300, sm_103a) and the built libtacaw.so")
    config.addinivalue_line("markers", "slow: long-running CPU test")


@pytest.fixture(scope="module", autouse=True)
def collected():
    """Every module starts with the garbage of the ones before it collected.  A test that catches an exception
    leaves its frame, and the device tensors in it, in a reference cycle; one that counts device memory
    would see them go whenever the collector happens to run."""
    gc.collect()
