import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)


def pytest_configure(config):
    config.addinivalue_line("markers", "gpu: needs a CUDA GPU (GB300, sm_103a)")


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


@pytest.fixture(scope="session")
def fake_cudart(tmp_path_factory):
    """Path of the stand-in for the CUDA runtime (fake_cudart.c), to preload in a child process."""
    import subprocess

    from paper_2412_15803_gb300 import build
    cuda = os.path.dirname(os.path.dirname(os.path.realpath(build.nvcc())))
    so = str(tmp_path_factory.mktemp("fake") / "libfake_cudart.so")
    subprocess.check_call(["gcc", "-O1", "-Wall", "-Werror", "-shared", "-fPIC", "-I", os.path.join(cuda, "include"),
                           "-o", so, os.path.join(ROOT, "tests", "fake_cudart.c")])
    build.build()
    return so
