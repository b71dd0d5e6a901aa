"""csrc/extents.h: the sizes and index walks that the kernels and their launches
share, compiled for the host.  No GPU."""
import ctypes
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2608_02474_gb300", "csrc")
WRAP = """
#include "extents.h"
extern "C" {
size_t stage_bytes(int n) { return key_stage_bytes(n); }
}
"""


@pytest.fixture(scope="module")
def ext(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no C++ compiler")
    d = tmp_path_factory.mktemp("extents")
    (d / "w.cpp").write_text(WRAP)
    subprocess.run([cxx, "-std=c++17", "-O1", "-shared", "-fPIC", "-I" + CSRC, str(d / "w.cpp"),
                    "-o", str(d / "w.so")], check=True)
    return ctypes.CDLL(str(d / "w.so"))


@pytest.mark.parametrize("n", [1, 2, 3, 4, 5, 7799, 7800, 10239, 51197, 51200])
def test_staged_keys_fit(ext, n):
    """The top-K kernels store keys as whole 16-byte groups at every multiple of four
    below n: the last one has to lie inside what the launch asks for."""
    ext.stage_bytes.restype = ctypes.c_size_t
    last_group = (n - 1) // 4
    assert 16 * (last_group + 1) <= ext.stage_bytes(n) < 16 * (last_group + 2)
    # and the launches ask for just that
    src = open(os.path.join(CSRC, "select.cu")).read()
    assert "const size_t key_bytes = key_stage_bytes(NT);" in src
    assert "key_stage_bytes(slice), st, keys" in src
