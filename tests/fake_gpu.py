"""The library's host paths without a GPU: its own objects, linked with a stand-in for the
CUDA runtime (fake_cudart.cpp) in which launches are written down instead of run and can be
made to fail. `fake_gpu` gives the controls; inside the test capi calls that build."""
import ctypes
import glob
import os
import subprocess

import pytest

from paper_2512_07311_gb300 import build as B
from paper_2512_07311_gb300 import capi

HERE = os.path.dirname(os.path.abspath(__file__))


class FakeGpu:
    def __init__(self, lib):
        self.lib = lib
        lib.fake_launch_kernel.restype = ctypes.c_char_p

    def reset(self, sms=152):
        self.lib.fake_reset(sms)

    def fail(self, kernel, code, skip=0, times=1):
        """The launches of kernels whose name holds `kernel` fail with `code`."""
        self.lib.fake_fail(kernel.encode(), skip, times, code)

    def launches(self):
        """(mangled kernel name, CTAs, device that was current) of every launch since reset."""
        return [(self.lib.fake_launch_kernel(i).decode(), self.lib.fake_launch_grid(i), self.lib.fake_launch_device(i))
                for i in range(self.lib.fake_launches())]


@pytest.fixture(scope="session")
def _fake_library(tmp_path_factory):
    B.build()
    objs = sorted(glob.glob(os.path.join(B.BUILD, "*.o")))
    if not objs:
        B.build(force=True)
        objs = sorted(glob.glob(os.path.join(B.BUILD, "*.o")))
    out = str(tmp_path_factory.mktemp("fake") / "librcs_fake.so")
    subprocess.run(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-Wl,-Bsymbolic", "-Wl,-z,defs", "-I", B._cuda_include(),
                    os.path.join(HERE, "fake_cudart.cpp"), *objs, "-o", out, "-lpthread"], check=True)
    return out


@pytest.fixture
def fake_gpu(_fake_library):
    real, capi._lib = capi._lib, None
    try:
        gpu = FakeGpu(capi.load(_fake_library))
        gpu.reset()
        yield gpu
    finally:
        capi._lib = real
