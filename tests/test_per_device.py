"""What belongs to a device is done once on each: the record itself, compiled for
the host and given made-up devices."""
import ctypes
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = r"""
#include "per_device.cuh"
static pdep::OncePerDevice once;
// result of the call and, in *acted, how often it acted
extern "C" int act(int device, int result, int* acted) {
  return once(device, [&] { ++*acted; return result; });
}
"""


def test_once_on_each_device(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    (tmp_path / "once.cpp").write_text(SRC)
    subprocess.run([cxx, "-std=c++17", "-shared", "-fPIC", "-I",
                    os.path.join(ROOT, "paper_1501_03141_gb300", "csrc"), "-o",
                    str(tmp_path / "once.so"), str(tmp_path / "once.cpp")], check=True)
    lib = ctypes.CDLL(str(tmp_path / "once.so"))

    def act(device, result=0):
        n = ctypes.c_int(0)
        return lib.act(device, result, ctypes.byref(n)), n.value

    assert act(0) == (0, 1) and act(0) == (0, 0)
    assert act(1) == (0, 1) and act(1) == (0, 0) and act(0) == (0, 0)
    assert act(2, 5) == (5, 1)  # a failure is not remembered
    assert act(2) == (0, 1) and act(2) == (0, 0)
    assert act(63) == (0, 1) and act(63) == (0, 0)
    assert act(64) == (0, 1) and act(64) == (0, 1)  # past the record: every time
