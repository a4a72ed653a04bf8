"""The build: the C library needs no PyTorch, and the native marshalling is a
file of the PyTorch and Python it was built against."""
import os
import shutil
import subprocess
import sys

import pytest
import torch

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PKG = "paper_2607_13093_gb300"


@pytest.fixture(scope="module")
def sph():
    from paper_2607_13093_gb300 import build_lib
    build_lib.build()
    from paper_2607_13093_gb300 import sph as m
    return m


def test_the_library_is_built_without_pytorch(sph, tmp_path):
    # a copy of the package with its objects, without library and marshalling
    shutil.copytree(os.path.join(ROOT, PKG), tmp_path / PKG, ignore=shutil.ignore_patterns("*.so"))
    shutil.copytree(os.path.join(ROOT, "include"), tmp_path / "include")
    code = (f"import sys; sys.modules['torch'] = None; from {PKG} import build_lib; "
            "print(build_lib.build())")
    r = subprocess.run([sys.executable, "-c", code], cwd=tmp_path, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    lib = tmp_path / PKG / "_lib" / "libsph.so"
    assert r.stdout.strip() == str(lib) and lib.exists()
    assert [p.name for p in lib.parent.glob("*.so")] == ["libsph.so"]


def test_another_pytorch_has_its_own_marshalling(sph, monkeypatch):
    from paper_2607_13093_gb300 import build_lib
    here = build_lib.fast_path()
    assert torch.__version__ in here and os.path.exists(here)
    assert sph._fast.__file__ == here
    monkeypatch.setattr(torch, "__version__", "0.0.1")
    there = build_lib.fast_path()
    assert there != here and not os.path.exists(there)
    with pytest.raises(RuntimeError, match="not built for this PyTorch"):
        sph._load_fast()
