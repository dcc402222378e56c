import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)


# The decode sizes of these modules run on the row-stream kernel by default, which stands in there for the kernels that they were
# written for: every test runs on both routes.
BOTH_ROUTES = ("test_gpu_gemm_ex", "test_zz_no_alloc")


def pytest_generate_tests(metafunc):
    if metafunc.module.__name__ in BOTH_ROUTES:
        metafunc.parametrize("decode_route", ["default", "others"], indirect=True)


@pytest.fixture(autouse=True)
def decode_route(request, monkeypatch):
    """"others": the row-stream kernel is never taken.  (The tests of the 4-bit decode kernel's default route need that, too.)"""
    if getattr(request, "param", None) == "others" or request.module.__name__ == "test_gpu_fp4":
        monkeypatch.setenv("BITDELTA_ROW", "0")


def pytest_configure(config):
    config.addinivalue_line("markers", "gpu: needs a CUDA device (sm_100a)")


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
