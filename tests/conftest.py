import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)


def pytest_configure(config):
    config.addinivalue_line("markers", "gpu: needs a CUDA device (runs the sm_100a kernels)")


def pytest_collection_modifyitems(config, items):
    try:
        import torch
        has_gpu = torch.cuda.is_available()
    except Exception:
        has_gpu = False
    if has_gpu:
        return
    skip = pytest.mark.skip(reason="no CUDA device")
    for item in items:
        if "gpu" in item.keywords:
            item.add_marker(skip)


@pytest.fixture
def group_size(request):
    """fsd_set_group_size for the test.  0: one kernel does a call whose logits fit on chip.  Else the streaming and finish kernels
    do it, in groups of that size or, where a row is too long for these, of the library's choice."""
    from paper_2502_20704_b200 import binding as fsd
    assert fsd.fsd_set_group_size(request.param) == 0
    yield request.param
    fsd.fsd_set_group_size(0)


def group_sizes(*sizes):
    """Marks that run a test, or a file's tests, once per group size."""
    return [pytest.mark.usefixtures("group_size"), pytest.mark.parametrize("group_size", sizes, indirect=True, ids=[f"groups{n}" for n in sizes])]
