import gc
import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)


def pytest_configure(config):
    config.addinivalue_line("markers", "gpu: needs a CUDA device (GB300, sm_103a)")
    config.addinivalue_line("markers", "slow: longer CPU test")


def pytest_runtest_setup(item):
    # A full collection in the middle of a test stops it for 16 to 40 ms once torch is loaded
    # (measured over a run), as long as two of the events that the admission tests expect to
    # find still running.  What is garbage goes now; the rest is not looked at again.
    gc.collect()
    gc.freeze()


@pytest.fixture(scope="session")
def oracle_lib():
    import oracle
    oracle.build()
    return oracle
