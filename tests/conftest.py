import gc
import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)


def pytest_configure(config):
    config.addinivalue_line("markers", "gpu: needs a CUDA GPU (GB300, sm_103a)")
    config.addinivalue_line("markers", "slow: long CPU oracle check")


def pytest_runtest_setup(item):
    # a caught exception and the frame that holds it form a cycle that keeps
    # the frame's tensors: collected at a defined time, not in the middle of a
    # test that counts device memory
    if item.get_closest_marker("gpu"):
        gc.collect()
