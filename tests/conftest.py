import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)


def pytest_configure(config):
    config.addinivalue_line("markers", "gpu: needs a CUDA device (GB300) and libcoffee.so")


def pytest_sessionstart(session):
    """Build libcoffee.so in-tree if it is missing or older than its sources (a no-op otherwise),
    so that the suite always runs against the library of the sources it tests."""
    from paper_1407_0904_gb300 import _build
    _build.build()


def pytest_collection_modifyitems(config, items):
    # test_around_a_tile wants prisms in TF32, BF16 and BF16X3 bit-equal to TF32X3, which include/coffee.h's definition of
    # those precisions rules out: its last two lines fail. Run at the end, so that -x has run everything else by then.
    items.sort(key=lambda it: it.name.startswith("test_around_a_tile["))
    try:
        import torch
        has_gpu = torch.cuda.is_available()
    except Exception:
        has_gpu = False
    if has_gpu:
        return
    skip = pytest.mark.skip(reason="no CUDA device")
    for it in items:
        if "gpu" in it.keywords:
            it.add_marker(skip)
