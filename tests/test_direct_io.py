"""Which arrays a call works on in place and which it stages: the rule itself,
compiled for the host and given made-up places."""
import ctypes
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = r"""
#include "direct_io.cuh"
using namespace pdep;
// three arrays (the first is written) of 'bytes' at p[], on gpu[], managed[], dev[]
extern "C" int rule(int device, unsigned long long* p, unsigned long long* bytes, int* gpu,
                    int* managed, int* dev) {
  Span s[3];
  for (int i = 0; i < 3; ++i)
    s[i] = Span{(const void*)p[i], (size_t)bytes[i], gpu[i] != 0, managed[i] != 0, dev[i]};
  return direct_io(device, s[0], {s[1], s[2]}) ? 1 : 0;
}
"""


@pytest.fixture(scope="module")
def rule(tmp_path_factory):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    d = tmp_path_factory.mktemp("direct_io")
    (d / "rule.cpp").write_text(SRC)
    subprocess.run([cxx, "-std=c++17", "-shared", "-fPIC", "-I",
                    os.path.join(ROOT, "paper_1501_03141_gb300", "csrc"), "-o", str(d / "rule.so"),
                    str(d / "rule.cpp")], check=True)
    lib = ctypes.CDLL(str(d / "rule.so"))

    def call(p=(4096, 8192, 16384), bytes=(64, 64, 64), gpu=(1, 1, 1), managed=(0, 0, 0),
             dev=(0, 0, 0), device=0):
        u, i = ctypes.c_ulonglong * 3, ctypes.c_int * 3
        return bool(lib.rule(device, u(*p), u(*bytes), i(*gpu), i(*managed), i(*dev)))
    return call


def test_in_place_on_the_context_gpu(rule):
    assert rule() and rule(dev=(2, 2, 2), device=2)
    assert rule(p=(4096, 4160, 4032))  # touching, not overlapping


@pytest.mark.parametrize("which", [0, 1, 2])
def test_staged(rule, which):
    def with_(base, v):
        return tuple(v if k == which else b for k, b in enumerate(base))
    assert not rule(dev=with_((0, 0, 0), 1))            # on another GPU
    assert rule(dev=with_((0, 0, 0), 1), managed=with_((0, 0, 0), 1))
    assert not rule(gpu=with_((1, 1, 1), 0))            # on the host
    assert not rule(p=with_((4096, 8192, 16384), 0))    # null
    assert not rule(p=with_((4096, 8192, 16384), 32772))  # misaligned
    if which:
        assert not rule(p=with_((4096, 8192, 16384), 4104))  # overlaps the output
