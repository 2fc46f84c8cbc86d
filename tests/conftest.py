import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)


def pytest_configure(config):
    config.addinivalue_line(
        "markers", "gpu: needs a CUDA GPU (sm_103a) and the built library")


def pytest_collection_modifyitems(config, items):
    # GPU tests are skipped, not failed, where no GPU is present so that the
    # CPU suite stays green; on a GPU machine they run.
    try:
        import torch
        has_gpu = torch.cuda.is_available()
    except Exception:  # pragma: no cover
        has_gpu = False
    if has_gpu:
        return
    skip = pytest.mark.skip(reason="no CUDA GPU in this process")
    for item in items:
        if "gpu" in item.keywords:
            item.add_marker(skip)


@pytest.fixture
def fused_rounds():
    """Every round the fused kernel covers runs on it: the stall hook is set
    to a stage no round has."""
    from paper_2608_02123_gb300 import pctree as P
    P.pctree_debug_stall_stage(1 << 20, 1_000_000_000)
    yield P
    P.pctree_debug_stall_stage(-1, 1_000_000_000)
