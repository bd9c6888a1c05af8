import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)


def pytest_configure(config):
    config.addinivalue_line("markers", "gpu: needs a GB300 GPU and the CUDA library")
    config.addinivalue_line("markers", "slow: CPU test that takes more than a few seconds")


def pytest_collection_finish(session):
    """Keeps the objects of the imports and the collection (some 200 000) out of later garbage collections: a
    full one took 70 ms, in the middle of whatever a test was timing."""
    import gc

    gc.collect()
    gc.freeze()
