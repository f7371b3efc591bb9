"""Shared pytest configuration: the ``gpu`` marker and the repo on sys.path."""
import contextlib
import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)


def pytest_configure(config):
    config.addinivalue_line(
        "markers", "gpu: needs a CUDA GPU (sm_103a) and the compiled library; "
        "run with -m gpu on a GB300")


@pytest.fixture
def swept():
    """``with swept():`` runs FP32 calls through the all-pairs sweep of the default
    rule where small ones would take the one launch without a sweep (profiling
    brackets the sweep, so it asks for one), and checks that they did."""
    @contextlib.contextmanager
    def run(handle=None):
        import paper_1402_4986_gb300 as idw
        idw.profile_enable(True, handle=handle)
        idw.profile_read(handle=handle)
        try:
            yield
            assert idw.profile_read(handle=handle)[1] > 0
        finally:
            idw.profile_enable(False, handle=handle)
    return run
