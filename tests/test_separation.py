"""The CUDA path and the oracle share no code, and the product path has no
CPU fallback.  No GPU.

- No file of the package (Python or CUDA) imports or includes the oracle, and
  the oracle imports nothing of the package.
- The seeded input generators (synth/) import neither.
- The binding fails loudly, before any compute, when the library is missing.
- It can be imported with a PyTorch that has no raw handle of the current stream.
"""
import ast
import glob
import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PKG = "paper_2608_02474_gb300"


def _imports(path):
    tree = ast.parse(open(path).read(), filename=path)
    out = set()
    for node in ast.walk(tree):
        if isinstance(node, ast.Import):
            out.update(a.name.split(".")[0] for a in node.names)
        elif isinstance(node, ast.ImportFrom) and node.module and node.level == 0:
            out.add(node.module.split(".")[0])
    return out


def _py(folder):
    return glob.glob(os.path.join(ROOT, folder, "**", "*.py"), recursive=True)


def test_package_never_imports_the_oracle():
    files = _py(PKG)
    assert files
    for f in files:
        assert "oracle" not in _imports(f), f
    for f in glob.glob(os.path.join(ROOT, PKG, "csrc", "*")):
        text = open(f, errors="replace").read()
        assert "oracle" not in text.lower(), f


def test_oracle_never_imports_the_package():
    for f in _py("oracle"):
        assert PKG not in _imports(f), f


def test_input_generators_import_neither_side():
    for f in _py("synth"):
        imps = _imports(f)
        assert "oracle" not in imps and PKG not in imps, f


def test_missing_library_fails_loudly(monkeypatch, tmp_path):
    from paper_2608_02474_gb300 import echocache as ec
    monkeypatch.setattr(ec, "_LIB", None)
    monkeypatch.setattr(ec, "LIB_PATH", str(tmp_path / "missing.so"))
    with pytest.raises(RuntimeError, match="missing"):
        ec.lib()


def test_import_without_the_raw_stream_name(monkeypatch):
    """A PyTorch built without CUDA lacks it: the import still works, and the handle comes
    from the Stream object."""
    import importlib.util

    import torch
    monkeypatch.delattr(torch._C, "_cuda_getCurrentRawStream", raising=False)
    spec = importlib.util.spec_from_file_location(
        "echocache_without_raw_stream", os.path.join(ROOT, PKG, "echocache.py"))
    ec = importlib.util.module_from_spec(spec)
    monkeypatch.setitem(sys.modules, spec.name, ec)
    spec.loader.exec_module(ec)

    class Stream:
        cuda_stream = 77

    monkeypatch.setattr(torch.cuda, "current_stream", lambda device=None: Stream)
    monkeypatch.setattr(ec, "_cur_device", lambda: 0)
    assert ec._stream() == 77 and ec._stream(Stream) == 77
