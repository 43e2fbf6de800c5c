import gc
import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)


def pytest_configure(config):
    config.addinivalue_line("markers", "gpu: needs a CUDA device (B200); parity tests through the C-ABI")


@pytest.fixture(scope="session")
def oracle():
    from oracle import photon_oracle
    photon_oracle.build()
    return photon_oracle


def pytest_runtest_setup(item):
    """The no-allocation tests compare the allocator's counters: tensors that earlier tests left in reference cycles (frames of
    tests that hold an exception) must not be freed in between."""
    if item.path.name == "test_zz_no_alloc.py":
        gc.collect()
