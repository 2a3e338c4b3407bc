"""The extension module belongs to one torch and one Python: it is rebuilt, and refused, when they are others."""
import os
import subprocess
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_rebuilt_for_another_torch(monkeypatch):
    import torch
    from paper_2107_06419_b200 import build
    build.build()
    calls = []
    monkeypatch.setattr(build, "build_binding", lambda: calls.append(1))
    monkeypatch.setattr(build, "build_library", lambda verbose=False: None)
    build.build()
    assert not calls
    monkeypatch.setattr(torch, "__version__", "2.0.0+another")
    build.build()
    assert calls


def test_refused_under_another_torch():
    code = "import torch; torch.__version__ = '2.0.0+another'; import paper_2107_06419_b200.api"
    r = subprocess.run([sys.executable, "-c", code], cwd=ROOT, capture_output=True, text=True, env={**os.environ, "PYTHONPATH": ROOT})
    assert r.returncode != 0 and "this is torch 2.0.0+another" in r.stderr and "paper_2107_06419_b200.build" in r.stderr
