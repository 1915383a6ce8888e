import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)


def pytest_configure(config):
    config.addinivalue_line("markers", "gpu: needs a CUDA GPU (sm_103a) and the built libgts")
    config.addinivalue_line("markers", "slow: long-running CPU case")


@pytest.fixture(scope="session")
def warp(tmp_path_factory):
    """The kernels' source built to run on the host (tests/warp_emulation.py): the executable and its folder."""
    from tests import warp_emulation
    path = str(tmp_path_factory.mktemp("warp"))
    exe = warp_emulation.build(path)
    if exe is None:
        pytest.skip("no g++ with the thread sanitizer")
    return exe, path
