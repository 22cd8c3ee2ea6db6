"""Shared pytest configuration: registers the `gpu` marker and puts the repo root on sys.path."""
import gc
import os
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)


def pytest_configure(config):
    config.addinivalue_line("markers", "gpu: test needs a CUDA device (run with -m gpu on a B200)")


def pytest_runtest_setup(item):
    """Handles that earlier tests left in reference cycles (a `pytest.raises` keeps the frames it caught) are freed here.  A free
    waits for the device, and inside a test of what waits for it and what does not, a collection changes the answer."""
    if item.get_closest_marker("gpu"):
        gc.collect()
