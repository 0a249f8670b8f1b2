"""The library linked against a CUDA runtime without a GPU (fake_cudart.cpp), for CPU tests of what the
host side launches: the fixture `fake` replaces the loaded library and offers the fake's controls;
`fake_torch` adds a torch whose device tensors lie in host memory."""
import contextlib
import ctypes
import glob
import os
import subprocess
import sys
import types

import pytest
import torch

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

    def give_up(self, kernel):
        """Launches of kernels with this in their name time out from now on (b"": none)."""
        self.dll.fake_give_up(kernel)

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


def _reset(f):
    f.set_device(0)
    f.fail_allocation(-1)
    f.give_up(b"")
    f.launched()


@pytest.fixture
def fake(_fake_library, monkeypatch):
    monkeypatch.setattr(gks, "_lib", None)
    gks.load_library(_fake_library.path)
    _reset(_fake_library)
    yield _fake_library
    _reset(_fake_library)


class FakeTorch:
    """torch with its "cuda" tensors in host memory, noting on which stream each is made and whose end
    a stream waits for."""

    class Stream:
        def __init__(self, torch, name):
            self.torch, self.name, self.cuda_stream = torch, name, 0

        def wait_stream(self, other):
            self.torch.waits.append((self.name, other.name))

    def __init__(self):
        self.made, self.waits = [], []
        self.cuda = types.SimpleNamespace(stream=self._on, current_stream=lambda: self.current,
                                          Stream=FakeTorch.Stream)
        self.current = self.Stream(self, "caller")

    def __getattr__(self, name):
        return getattr(torch, name)

    @contextlib.contextmanager
    def _on(self, stream):
        before, self.current = self.current, stream
        yield
        self.current = before

    def _make(self, fn, size, dtype, device):
        self.made.append(self.current.name)
        return _Tensor(fn(size, dtype=dtype))

    def empty(self, size, dtype=None, device=None):
        return self._make(torch.empty, size, dtype, device)

    def zeros(self, size, dtype=None, device=None):
        return self._make(torch.zeros, size, dtype, device)


class _Tensor:
    def __init__(self, t):
        self.t, self.streams = t, []

    def record_stream(self, s):
        self.streams.append(s.name)

    def __rmul__(self, other):
        return other * self.t

    def __getattr__(self, name):
        return getattr(self.t, name)


@pytest.fixture
def fake_torch(fake, monkeypatch):
    t = FakeTorch()
    monkeypatch.setitem(sys.modules, "torch", t)
    return t
