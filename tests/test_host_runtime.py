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
OUT_OF_MEMORY, ILLEGAL_ADDRESS = 2, 700  # cudaErrorMemoryAllocation, cudaErrorIllegalAddress


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
    ps.ps_plan_destroy(ps.ps_plan_create(ps.make_config(8)))  # gives back what an earlier call kept
    assert f.lib.fake_live() == 0
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


NORM = dict(mean=np.zeros(5), std=np.ones(5), s_tau=1.0, s_A=1.0)


def _attach(fake, plan):
    fake.ps.ps_plan_set_closure(plan, np.zeros(fake.ps.MLP_NPARAM, np.float32).ctypes.data, NORM)


@pytest.mark.parametrize("nth", range(1, 9))
def test_a_closure_that_could_not_be_attached_can_be_attached_later(fake, nth):
    """An allocation that fails leaves nothing behind, and the next call
    allocates every buffer."""
    cfg = fake.ps.make_config(32, nu=1e-3)
    whole, again = (fake.ps.ps_plan_create(cfg) for _ in range(2))
    before = fake.lib.fake_live()
    _attach(fake, whole)
    need = fake.lib.fake_live() - before
    fake.fail("cudaMalloc", nth, OUT_OF_MEMORY)
    with pytest.raises(fake.ps.PsError) as e:
        _attach(fake, again)
    assert e.value.status == fake.ps.PS_ERR_OOM
    assert fake.lib.fake_live() == before + need
    _attach(fake, again)
    assert fake.lib.fake_live() == before + 2 * need
    for plan in (whole, again):
        fake.ps.ps_plan_destroy(plan)
    assert fake.lib.fake_live() == 0
