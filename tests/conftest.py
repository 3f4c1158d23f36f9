import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)


def pytest_configure(config):
    config.addinivalue_line("markers", "gpu: needs a CUDA device (GB300, sm_103a)")
    config.addinivalue_line("markers", "slow: longer-running check")


def pytest_collection_modifyitems(items):
    # The serving tests go first.  Their stream of requests 10 ms apart has to
    # overlap, and a request of these sizes takes 1 to 2 ms: it is the first
    # ones, while a fresh process loads the library's kernels, that do.
    items.sort(key=lambda item: item.path.name != "test_gpu_serve.py")
