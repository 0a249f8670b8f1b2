"""The library linked against a CUDA runtime without a GPU (fake_cudart.cpp), for CPU tests of what the
host side launches: the fixture `fake` replaces the loaded library and offers the fake's controls."""
import ctypes
import glob
import os
import subprocess

import pytest

from paper_2412_16845_gb300 import build as gbuild
from paper_2412_16845_gb300 import gks

HERE = os.path.dirname(os.path.abspath(__file__))


class Fake:
    def __init__(self, path):
        self.path = path
        self.dll = ctypes.CDLL(path)
        self.dll.fake_launched.restype = ctypes.c_char_p

    def set_device(self, d):
        self.dll.fake_set_device(d)

    def fail_allocation(self, after):
        """The allocation after `after` more fails (-1: none)."""
        self.dll.fake_fail_allocation(after)

    def launched(self):
        """Names of the kernels launched since the last call."""
        names = self.dll.fake_launched().decode().split()
        self.dll.fake_clear()
        return names


@pytest.fixture(scope="session")
def _fake_library(tmp_path_factory):
    gbuild.build()
    inc = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(gbuild._nvcc()))), "include")
    out = str(tmp_path_factory.mktemp("fake") / "libgks_fake.so")
    objs = sorted(glob.glob(os.path.join(gbuild.BUILD, "*.o")))
    r = subprocess.run(["g++", "-std=c++17", "-O1", "-fPIC", "-shared", "-Wl,-Bsymbolic", "-I", inc,
                        os.path.join(HERE, "fake_cudart.cpp"), *objs, "-o", out],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return Fake(out)


@pytest.fixture
def fake(_fake_library, monkeypatch):
    monkeypatch.setattr(gks, "_lib", None)
    gks.load_library(_fake_library.path)
    _fake_library.set_device(0)
    _fake_library.fail_allocation(-1)
    _fake_library.launched()
    yield _fake_library
    _fake_library.set_device(0)
    _fake_library.fail_allocation(-1)
