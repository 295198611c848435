"""The library linked with tests/fake_cuda.cpp in place of the CUDA runtime:
kernels do nothing, and allocations, devices and launches fail as a test says.
For host code whose faults must not be run on a GPU."""
import ctypes
import os
import shutil
import subprocess

import pytest

from paper_1912_08453_gb300 import build, ccpm

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="session")
def fake_library(tmp_path_factory):
    build.build()
    path = str(tmp_path_factory.mktemp("fake") / "libccpm_fake.so")
    objs = [os.path.join(build.BUILD, s + ".o") for s in build.SOURCES]
    if not all(os.path.exists(o) for o in objs):
        pytest.skip("the library's objects are not here")
    include = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(build._nvcc()))), "include")
    # -Bsymbolic: these definitions serve the library, whatever runtime the process has loaded
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-Wl,-Bsymbolic", "-I", include,
                    os.path.join(HERE, "fake_cuda.cpp"), *objs, "-o", path], check=True)
    return path


@pytest.fixture()
def fake(fake_library, tmp_path, monkeypatch):
    """The fake's controls; ccpm calls the fake library meanwhile (a copy of its
    own for each test: nothing it keeps per process is left from another).  A test
    closes what it made, so that no handle of the fake reaches the real library."""
    path = shutil.copy(fake_library, tmp_path)
    monkeypatch.setattr(ccpm, "_LIB_PATH", path)
    monkeypatch.setattr(ccpm, "lib", ccpm._load())
    f = ctypes.CDLL(path)
    f.fake_limit.argtypes = [ctypes.c_size_t]
    f.fake_fail_at.argtypes = [ctypes.c_long]
    f.fake_calls.argtypes = [ctypes.c_char_p]
    for name in ("fake_allocs", "fake_bad", "fake_calls"):
        getattr(f, name).restype = ctypes.c_long
    f.fake_in_use.restype = f.fake_peak.restype = ctypes.c_size_t
    f.fake_reset()
    yield f
    assert f.fake_in_use() == 0, "device memory left behind"
