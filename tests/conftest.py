import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)


def pytest_configure(config):
    config.addinivalue_line("markers", "gpu: needs a CUDA GPU (GB300, sm_103a) and the built library")
    config.addinivalue_line("markers", "slow: long-running CPU test")


def _has_gpu():
    try:
        import torch
        return torch.cuda.is_available()
    except Exception:
        return False


def pytest_collection_modifyitems(config, items):
    if _has_gpu():
        return
    skip = pytest.mark.skip(reason="no CUDA device")
    for item in items:
        if "gpu" in item.keywords:
            item.add_marker(skip)


@pytest.fixture(scope="module", autouse=True)
def _tuning_table_as_shipped():
    """Entries that a module's tests add to the process-wide tuning table do
    not reach the next module's."""
    yield
    package = sys.modules.get("paper_1905_03136_gb300._lib")
    if package is not None and package._lib is not None:
        path = os.environ.get("TSM_TUNE_FILE") or package.DEFAULT_TABLE
        if os.path.exists(path):
            package._lib.tsm_clear_tuning()
            package._lib.tsm_load_tuning(path.encode())
