import gc
import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)


def pytest_configure(config):
    config.addinivalue_line("markers", "gpu: needs a CUDA GPU (runs the sm_103a library)")
    config.addinivalue_line("markers", "slow: long-running CPU test")


def pytest_collection_modifyitems(config, items):
    # GPU tests are skipped (not failed) when no GPU is present, unless the
    # caller explicitly selected them with -m gpu, in which case a missing GPU
    # or library must fail loudly.
    try:
        import torch
        have_gpu = torch.cuda.is_available()
    except Exception:  # pragma: no cover
        have_gpu = False
    markexpr = config.getoption("-m") or ""
    if have_gpu or ("gpu" in markexpr and "not gpu" not in markexpr):
        return
    skip = pytest.mark.skip(reason="no CUDA GPU in this environment")
    for it in items:
        if "gpu" in it.keywords:
            it.add_marker(skip)


@pytest.fixture(autouse=True)
def _no_garbage_from_earlier_cases(request):
    # The allocator checks compare torch.cuda.memory_allocated() around library calls.  An earlier case's
    # pytest.raises keeps its frame, and the tensors in it, in a reference cycle that the collector frees whenever it
    # next runs, also between the two readings: it runs here instead.
    if request.module.__name__ == "test_zz_no_alloc":
        gc.collect()
