import gc
import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)


def pytest_configure(config):
    config.addinivalue_line("markers", "gpu: needs a CUDA GPU (GB300, sm_103a) and the built libgbrt.so")


@pytest.fixture(scope="session")
def oracle():
    import oracle as O
    O.lib()
    return O


def pytest_runtest_setup(item):
    # an earlier test's traceback can hold device tensors in a cycle; collected
    # in the middle of a test that counts allocations, they would show there
    if item.get_closest_marker("gpu"):
        gc.collect()
