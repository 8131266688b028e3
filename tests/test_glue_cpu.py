"""How the torch side of the modules gets loaded: by the first call, from a build of the present sources."""
import importlib
import os
import subprocess
import sys

import pytest

from paper_2405_03133_b200 import build

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_importing_the_modules_loads_no_library():
    """Only a call needs the CUDA library; without one it says so, and a CPU tensor is refused before that."""
    code = """
import torch
from paper_2405_03133_b200 import LoryError, layer
m = layer.LoryMoE(8, 8, 2, T=4, device="cpu")
for call in (lambda: m(torch.zeros(1, 4, 8, dtype=torch.bfloat16)), layer._glue):
    try:
        call()
    except RuntimeError as e:
        print(type(e).__name__)
assert issubclass(LoryError, RuntimeError)
"""
    env = dict(os.environ, LORY_LIBRARY=os.path.join(ROOT, "no_such_library.so"))
    out = subprocess.run([sys.executable, "-c", code], cwd=ROOT, env=env, capture_output=True, text=True, timeout=300)
    assert out.stdout.split() == ["RuntimeError", "LoryError"], out.stderr


@pytest.mark.parametrize("content,current", [(None, False), (b"lory-glue-0123", False), ("tag", True)])
def test_a_glue_of_other_sources_is_not_taken(tmp_path, monkeypatch, content, current):
    glue = tmp_path / "_torch_glue.so"
    if content is not None:
        glue.write_bytes(b"\x7fELF.." + (build.glue_tag().encode() if content == "tag" else content) + b"..")
    monkeypatch.setattr(build, "GLUE", str(glue))
    assert build.glue_is_current() == current
    built = []
    monkeypatch.setattr(build.subprocess, "run", lambda cmd, **kw: built.append(cmd) or subprocess.CompletedProcess(cmd, 1, "", ""))
    if current:
        assert build.build_glue() == str(glue)
    else:
        with pytest.raises(RuntimeError):    # the compiler stands in here: that it was asked is the point
            build.build_glue()
    assert bool(built) != current


def test_the_tag_follows_every_source(tmp_path, monkeypatch):
    tag = build.glue_tag()
    changed = tmp_path / "glue.cpp"
    changed.write_bytes(open(build.GLUE_SRC, "rb").read() + b"// changed")
    monkeypatch.setattr(build, "GLUE_SRC", str(changed))
    assert build.glue_tag() != tag


def test_the_first_call_asks_for_a_current_glue(monkeypatch):
    """The loader looks at the file before it imports it: a module that has been imported cannot be replaced."""
    from paper_2405_03133_b200 import layer
    asked = []

    class Module:
        @staticmethod
        def bind(path, check):
            asked.append("bind")

    monkeypatch.setattr(layer, "_module", None)
    monkeypatch.setattr(layer._lory, "load", lambda: asked.append("library"))
    monkeypatch.setattr(build, "build_glue", lambda force=False: asked.append("build"))
    monkeypatch.setattr(importlib, "import_module", lambda *a: asked.append("import") or Module)
    assert layer._glue() is Module and layer._glue() is Module
    assert asked == ["library", "build", "import", "bind"]
