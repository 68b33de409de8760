import gc
import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)


def pytest_configure(config):
    config.addinivalue_line("markers", "gpu: needs a CUDA GPU (GB300, sm_103a)")


def pytest_sessionstart(session):
    # the library and the oracle are built in-tree; make sure they exist
    so = os.path.join(ROOT, "paper_1302_6189_gb300", "_lib", "libmdfft.so")
    if not os.path.exists(so):
        import __graft_entry__
        __graft_entry__.build()


def pytest_collection_modifyitems(config, items):
    try:
        import torch
        have_gpu = torch.cuda.is_available()
    except Exception:
        have_gpu = False
    if have_gpu:
        return
    skip = pytest.mark.skip(reason="no CUDA GPU on this host")
    for item in items:
        if "gpu" in item.keywords:
            item.add_marker(skip)


def pytest_runtest_setup(item):
    # the no-allocation test compares torch's allocated bytes around its calls:
    # tensors that an earlier test's exception traceback still holds in a
    # reference cycle must not be collected in between
    if "no_alloc" in item.nodeid:
        gc.collect()
