import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)


@pytest.fixture
def kernels():
    """kernels(call): the names of this library's kernels that call() launched
    (which of several paths a call took; all of them give the same bits)."""
    from paper_2607_29221_gb300 import mosaic as M

    def run(call):
        M.mosaic_kernel_times(reset=True)
        M.mosaic_kernel_timing(True)
        try:
            call()
            M.mosaic_device_status()
            return {name.split(":")[1] for name in M.mosaic_kernel_times(reset=True)}
        finally:
            M.mosaic_kernel_timing(False)
    return run


def pytest_configure(config):
    config.addinivalue_line("markers", "gpu: needs a GB300 (runs the CUDA library)")
    config.addinivalue_line("markers", "slow: long-running case")
