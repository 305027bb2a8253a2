import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)


def pytest_configure(config):
    config.addinivalue_line("markers", "gpu: needs a CUDA GPU (GB300) and runs the CUDA kernels")


@pytest.fixture(scope="session")
def cuda_lib():
    """Builds (if needed) and loads libmemplan.so; GPU tests fail loudly without CUDA."""
    import torch

    assert torch.cuda.is_available(), "GPU test run without a CUDA device"
    from paper_2203_00448_gb300 import build
    from paper_2203_00448_gb300 import _lib

    build.build()
    return _lib.load()


ROUTES = ("first", "walk", "phases", "general", "grid-flow", "grid-phases", "breadth-comp", "breadth-phases",
          "breadth-tensor")  # mp::TestRoute


@pytest.fixture
def routes(cuda_lib):
    """The package on a test build of the library that counts the traces each
    placement route takes: yields a function that returns {route: traces} since
    its last call, routes that took none left out."""
    import ctypes

    from paper_2203_00448_gb300 import _lib, build

    path = build.build_test_hooks()
    plain, _lib._lib = _lib._lib, None
    try:
        lib = _lib.load(path)
        counts = (ctypes.c_uint32 * len(ROUTES))()

        def read():
            assert lib.mp_test_routes(counts) == 0
            return {r: c for r, c in zip(ROUTES, counts) if c}

        read()
        yield read
    finally:
        _lib._lib = plain
