import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)


def pytest_configure(config):
    config.addinivalue_line("markers", "gpu: needs a CUDA device (run on the B200 box)")


def pytest_collection_modifyitems(config, items):
    try:
        import torch
        has_gpu = torch.cuda.is_available()
    except Exception:  # pragma: no cover
        has_gpu = False
    if has_gpu:
        return
    skip = pytest.mark.skip(reason="no CUDA device")
    for item in items:
        if "gpu" in item.keywords:
            item.add_marker(skip)


@pytest.fixture(autouse=True, scope="session")
def copy_streams_made(request):
    """The first host-buffer call of a process makes the copy streams, events and pinned words that later ones share: mostly 2.5 ms, but 44 ms in one
    process of four on a busy host.  Tests that time such calls mean the calls."""
    if not any("gpu" in item.keywords for item in request.session.items):
        return
    import torch
    if not torch.cuda.is_available():
        return
    from paper_2511_04002_b200 import binding as B
    T, H = 1024, 4096                                          # two parts
    plan = B.Plan(torch.float16, H, T, 6.0, [2, 4, 8], 0.2)
    blob, ws = plan.alloc(T)
    x = torch.zeros((T, H), dtype=torch.float16).pin_memory()
    blob_host = torch.empty(blob.numel(), dtype=torch.uint8).pin_memory()
    plan.encode_host(x, blob_host, torch.empty_like(x, device="cuda"), blob, ws)
