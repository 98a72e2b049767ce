import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)


def _ensure_library_is_built():
    """The package refuses its calls without libmqgrad.so and the binding for this interpreter and
    torch (there is no fallback path), so a checkout that lacks either builds it here once; nvcc
    cross-compiles without a GPU.  (Files that are older than their sources are left alone: a copy
    of a built tree need not keep the times.)"""
    import importlib.util
    spec = importlib.util.spec_from_file_location("_mqg_build", os.path.join(ROOT, "paper_1804_08066_b200", "build.py"))
    mod = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(mod)
    if not os.path.exists(mod.LIB) or not os.path.exists(mod.binding_path()):
        mod.build()


_ensure_library_is_built()


def pytest_configure(config):
    config.addinivalue_line("markers", "gpu: needs a CUDA device (run on a B200)")


def pytest_collection_modifyitems(config, items):
    try:
        import torch
        have = torch.cuda.is_available()
    except Exception:  # pragma: no cover
        have = False
    if have:
        return
    skip = pytest.mark.skip(reason="no CUDA device")
    for it in items:
        if "gpu" in it.keywords:
            it.add_marker(skip)
