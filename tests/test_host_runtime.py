"""The library's host code against a CUDA runtime that returns errors on demand
(tests/fake_cudart.cpp, linked with the library's own objects): what a call
reports, keeps and gives back when an allocation or a synchronisation fails.
No GPU is used and no kernel runs."""

import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1808_01309_gb300", "csrc")
ILLEGAL_ADDRESS = 700  # cudaErrorIllegalAddress


@pytest.fixture(scope="module")
def host_lib(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    from paper_1808_01309_gb300 import build
    build.build()
    objs = [os.path.join(build.BUILD, f[:-3] + ".o") for f in sorted(os.listdir(CSRC)) if f.endswith(".cu")]
    if not all(map(os.path.exists, objs)):
        build.build(force=True)
    cuda = os.path.dirname(os.path.dirname(os.path.realpath(build._nvcc())))
    out = str(tmp_path_factory.mktemp("host") / "libps_host.so")
    subprocess.run([cxx, "-std=c++17", "-O1", "-Wall", "-Werror", "-fPIC", "-shared", "-Wl,-Bsymbolic",
                    "-I", os.path.join(cuda, "include"), os.path.join(ROOT, "tests", "fake_cudart.cpp"), *objs,
                    "-lpthread", "-o", out], check=True)
    return out


class Fake:
    """The library over the fake runtime."""

    def __init__(self, ps, lib):
        self.ps, self.lib = ps, lib
        lib.fake_live.restype = lib.fake_peak.restype = ctypes.c_size_t
        lib.fake_budget.argtypes = [ctypes.c_size_t]
        lib.fake_launches.restype = ctypes.c_char_p

    def fail(self, call, nth, code):
        self.lib.fake_fail(call.encode(), nth, code)

    def sample(self, nd=32, nl=16, kc=5):
        u = np.zeros((3, nd, nd, nd // 2 + 1), np.complex64)
        out = [np.zeros((nl ** 3, k), np.float32) for k in (5, 9, 6)]
        self.ps.ps_les_training_sample(nd, u.ctypes.data, nl, kc, None, *(o.ctypes.data for o in out))


@pytest.fixture
def fake(host_lib, monkeypatch):
    from paper_1808_01309_gb300 import ps
    monkeypatch.setattr(ps, "_lib", None)
    f = Fake(ps, ps.load(host_lib))
    f.lib.fake_reset()
    yield f
    f.lib.fake_reset()


def test_a_failure_seen_at_the_synchronisation_of_a_sample_is_reported(fake):
    fake.sample()
    fake.fail("cudaStreamSynchronize", 1, ILLEGAL_ADDRESS)
    with pytest.raises(fake.ps.PsError, match="ps_les_training_sample") as e:
        fake.sample()
    assert e.value.status == fake.ps.PS_ERR_CUDA
    assert fake.lib.fake_live() == 0  # no block is kept after a failure
    fake.lib.fake_reset()  # (a real illegal address ends the context)
    fake.sample()
