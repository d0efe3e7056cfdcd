"""When the binding's native module is rebuilt, and what its absence says (no GPU needed)."""
import os
import shutil
import subprocess
import sys

import torch

from paper_2607_17979_b200 import build

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_a_binding_built_for_another_torch_is_stale(monkeypatch, tmp_path):
    copy = tmp_path / "_binding.so"
    shutil.copy(build.BINDING, copy)
    os.utime(copy)                          # newer than every source
    monkeypatch.setattr(build, "BINDING", str(copy))
    built = []
    monkeypatch.setattr(build, "is_stale", lambda: False)
    monkeypatch.setattr(build, "_build_binding", lambda: built.append(1))
    build.build()
    assert not built
    monkeypatch.setattr(torch, "__version__", torch.__version__ + ".post1")
    build.build()
    assert built == [1]


def test_import_without_the_binding_names_the_build_command(tmp_path):
    package = tmp_path / "paper_2607_17979_b200"
    package.mkdir()
    for name in ("__init__.py", "api.py", os.path.basename(build.LIB)):
        shutil.copy(os.path.join(build.HERE, name), package / name)
    r = subprocess.run([sys.executable, "-c", "import paper_2607_17979_b200.api"], cwd=tmp_path, capture_output=True, text=True,
                       env={k: v for k, v in os.environ.items() if k != "PYTHONPATH"})
    assert r.returncode != 0 and "ImportError" in r.stderr
    assert "python -m paper_2607_17979_b200.build" in r.stderr.strip().splitlines()[-1]
