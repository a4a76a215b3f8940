import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)


@pytest.fixture
def kernels():
    """kernels(call): the names of this library's kernels that call() launched
    (which of several paths a call took; all of them give the same bits), as a
    set, or by the entry point's role as {role: set}."""
    from paper_2607_29221_gb300 import mosaic as M

    def run(call, by_role=False):
        M.mosaic_kernel_times(reset=True)
        M.mosaic_kernel_timing(True)
        try:
            call()
            M.mosaic_device_status()
            names = [name.split(":") for name in M.mosaic_kernel_times(reset=True)]
            if by_role:
                return {role: {k for r, k in names if r == role} for role, _ in names}
            return {k for _, k in names}
        finally:
            M.mosaic_kernel_timing(False)
    return run


def pytest_configure(config):
    config.addinivalue_line("markers", "gpu: needs a GB300 (runs the CUDA library)")
    config.addinivalue_line("markers", "slow: long-running case")
