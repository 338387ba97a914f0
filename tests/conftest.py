import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)


def pytest_configure(config):
    config.addinivalue_line("markers", "gpu: needs a CUDA device (B200) and the built library")


def pytest_collection_modifyitems(config, items):
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


@pytest.fixture(scope="module", params=["clusters", "chain"])
def ctx(request):
    """A context that takes the one-launch form of short calls, and one whose every call goes through the kernels of long
    ones: most sizes that a test can afford are short, and both kinds of kernels serve the same entry points."""
    from paper_2506_08889_b200 import binding
    with pytest.MonkeyPatch.context() as mp:
        mp.setenv("SEER_STEP_CLUSTERS", "1" if request.param == "clusters" else "0")      # read when a context is created
        c = binding.Context(0)
    c.one_launch = request.param == "clusters"
    yield c
    c.close()
