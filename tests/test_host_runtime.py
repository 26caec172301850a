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


class Calls:
    """Calls that allocate device memory, each on objects made beforehand."""

    def __init__(self, fake):
        self.ps, self.fake, self.made = fake.ps, fake, []
        self.n = 32
        self.u = np.zeros((3, 32, 32, 17), np.complex64)
        self.f = np.ones_like(self.u)
        self.vec, self.loss = np.zeros(fake.ps.MLP_NPARAM, np.float32), np.zeros(1)

    def plan(self):
        self.made.append((self.ps.ps_plan_destroy, self.ps.ps_plan_create(self.ps.make_config(self.n, nu=1e-3))))
        return self.made[-1][1]

    def close(self):
        for destroy, handle in reversed(self.made):
            destroy(handle)
        self.made = []

    def prepare(self, name):
        """The objects of one call; returns the call."""
        ps, u, vec = self.ps, self.u.ctypes.data, self.vec.ctypes.data
        if name == "plan":
            return self.plan
        if name in ("closure", "closure gradient", "closure transfer"):
            p = self.plan()
            if name == "closure":
                return lambda: _attach(self.fake, p)
            _attach(self.fake, p)
            if name == "closure gradient":
                return lambda: ps.ps_plan_closure_grad(p, vec, u, self.f.ctypes.data, vec, self.loss.ctypes.data)
            return lambda: ps.ps_plan_closure_grad_transfer(p, vec, u, np.zeros(8), vec, self.loss.ctypes.data)
        if name in ("host step", "host step, copy engines"):
            p = self.plan()
            ps.ps_plan_set_host_mode(p, ps.HOST_AUTO if name == "host step" else ps.HOST_CUBE_CE)
            return lambda: ps.ps_rk_step_host(p, u, 1e-3)
        if name == "slab":
            cfg = ps.make_config(self.n, nu=1e-3, forcing=self.f.ctypes.data)
            return lambda: self.made.append((ps.ps_slab_destroy, ps.ps_slab_create(cfg, 0, 6, 0, 16)))
        if name == "backward transform":
            return lambda: ps.ps_fft_c2r(self.n, 3, u, np.zeros((3, 32, 32, 32), np.float32).ctypes.data)
        if name == "sample":
            return lambda: self.fake.sample(64, 32, 10)
        e = ps.ps_ensemble_create([ps.make_config(self.n, nu=1e-3) for _ in range(2)])
        self.made.append((ps.ps_ensemble_destroy, e))
        states = [self.u.ctypes.data] * 2
        if name == "ensemble tuning":
            return lambda: ps.ps_ensemble_tune(e, states, 1e-3)
        mode = ps.ENS_PERSISTENT if name == "persistent ensemble" else ps.ENS_BATCHED
        return lambda: ps.ps_ensemble_rk_steps(e, states, 1e-3, 0.0, 2, mode)


@pytest.mark.parametrize("name", ["plan", "closure", "closure gradient", "closure transfer", "host step",
                                  "host step, copy engines", "slab", "backward transform", "sample",
                                  "persistent ensemble", "batched ensemble", "ensemble tuning"])
def test_a_call_that_fits_without_the_kept_scratch_fits_with_it(fake, name):
    """Memory for a call, and no more: the block that a training sample left is
    given back to it."""
    calls = Calls(fake)
    call = calls.prepare(name)
    fake.lib.fake_reset()
    call()
    need = fake.lib.fake_peak()
    calls.close()
    fake.ps.ps_plan_destroy(fake.ps.ps_plan_create(fake.ps.make_config(8)))
    assert fake.lib.fake_live() == 0
    call = calls.prepare(name)
    before = fake.lib.fake_live()
    fake.sample()
    assert fake.lib.fake_live() > before  # a block is kept
    fake.lib.fake_budget(need)
    try:
        call()
    finally:
        calls.close()


@pytest.mark.parametrize("nth", [1, 2])
def test_a_persistent_ensemble_recovers_from_a_work_list_that_did_not_fit(fake, nth):
    calls = Calls(fake)
    call = calls.prepare("persistent ensemble")
    e, states = calls.made[-1][1], [calls.u.ctypes.data] * 2
    call()  # two steps: a list of that size
    fake.fail("cudaMalloc", nth, OUT_OF_MEMORY)
    with pytest.raises(fake.ps.PsError) as err:
        fake.ps.ps_ensemble_rk_steps(e, states, 1e-3, 0.0, 5, fake.ps.ENS_PERSISTENT)
    assert err.value.status == fake.ps.PS_ERR_OOM
    fake.lib.fake_reset()
    call()
    calls.close()
    assert fake.lib.fake_live() == 0


def test_a_host_step_recovers_from_a_zero_buffer_that_did_not_fit(fake):
    calls = Calls(fake)
    call = calls.prepare("host step, copy engines")
    fake.fail("cudaMalloc", 2, OUT_OF_MEMORY)  # (the first is the device state)
    with pytest.raises(fake.ps.PsError) as err:
        call()
    assert err.value.status == fake.ps.PS_ERR_OOM
    fake.lib.fake_reset()
    call()
    calls.close()
    assert fake.lib.fake_live() == 0


def _launches(fake, captured):
    """(kernel, grid, block, shared memory) of the passes launched in or out of a capture."""
    rows = [line.rsplit(" ", 1) for line in fake.lib.fake_launches().decode().splitlines()]
    kinds = ("k_zinv", "k_yinv", "k_xpass", "k_yfwd", "k_zfwd")
    return [what for what, flag in rows if flag == str(int(captured)) and any(k in what for k in kinds)]


@pytest.mark.parametrize("sizes", [(32, 32), (64,) * 3, (64,) * 12, (128, 64, 128, 64)], ids=str)
def test_the_ensemble_tuner_times_the_kernels_that_the_graph_runs(fake, sizes):
    """Where the tuner keeps the default shapes, what it timed plan by plan is
    what the graph launches, and a second tuning times the same again.  A branch
    per member is among the branch counts."""
    ps = fake.ps
    e = ps.ps_ensemble_create([ps.make_config(n, nu=1e-3) for n in sizes])
    states = [np.zeros((3, n, n, n // 2 + 1), np.complex64) for n in sizes]
    ptrs = [s.ctypes.data for s in states]
    timed = []
    for _ in range(2):
        fake.lib.fake_reset()
        tuning = ps.ps_ensemble_tune(e, ptrs, 1e-3)
        assert tuning["branches"] == len(sizes) and not any(tuning["xrpc"].values())
        timed.append(_launches(fake, False))
    assert timed[0] == timed[1]
    fake.lib.fake_reset()
    ps.ps_ensemble_rk_steps(e, ptrs, 1e-3, 0.0, 1, ps.ENS_GRAPH)
    run = set(_launches(fake, True))
    assert len(run) == 5 * len(set(sizes)) and run <= set(timed[0])
    # and a member stepped alone afterwards takes the launches of a plan alone
    fake.lib.fake_reset()
    ps.ps_ensemble_rk_steps(e, ptrs, 1e-3, 0.0, 1, ps.ENS_SEQUENTIAL)
    alone = set(_launches(fake, False))
    fake.lib.fake_reset()
    for n, s in zip(sizes, ptrs):
        plan = ps.ps_plan_create(ps.make_config(n, nu=1e-3))
        ps.ps_rk_step(plan, s, 1e-3)
        ps.ps_plan_destroy(plan)
    assert alone == set(_launches(fake, False))
    ps.ps_ensemble_destroy(e)


def _tables(fake):
    """Launches of the integrating-factor tables out of a capture."""
    return sum("k_if_tables" in line and line.endswith(" 0") for line in fake.lib.fake_launches().decode().splitlines())


def test_a_replayed_graph_leaves_the_tables_of_its_own_step(fake):
    """A graph computes the factor tables of its dt at every replay: a single
    step with another dt after it needs its own again."""
    ps = fake.ps
    plan, u = ps.ps_plan_create(ps.make_config(32, nu=1e-3)), np.zeros((3, 32, 32, 17), np.complex64).ctypes.data
    ps.ps_rk_steps(plan, u, 1e-3, 0.0, 2)
    ps.ps_rk_step(plan, u, 2e-3)
    ps.ps_rk_steps(plan, u, 1e-3, 0.0, 2)  # replayed
    fake.lib.fake_reset()
    ps.ps_rk_step(plan, u, 2e-3)
    assert _tables(fake) == 1
    ps.ps_rk_step(plan, u, 2e-3)
    assert _tables(fake) == 1
    ps.ps_plan_destroy(plan)


@pytest.mark.parametrize("mode", ["ENS_GRAPH", "ENS_PERSISTENT", "ENS_BATCHED"])
def test_a_replayed_ensemble_graph_leaves_the_tables_of_its_own_step(fake, mode):
    calls = Calls(fake)
    calls.prepare("persistent ensemble")
    ps, e, states = fake.ps, calls.made[-1][1], [calls.u.ctypes.data] * 2

    def step(dt, m):
        ps.ps_ensemble_rk_steps(e, states, dt, 0.0, 1, getattr(ps, m))

    for dt, m in ((1e-3, mode), (2e-3, "ENS_SEQUENTIAL"), (1e-3, mode)):
        step(dt, m)
    fake.lib.fake_reset()
    step(2e-3, "ENS_SEQUENTIAL")
    assert _tables(fake) == 2
    calls.close()


@pytest.mark.parametrize("call", ["cudaGraphInstantiate", "cudaGraphLaunch"])
def test_tables_of_a_graph_that_did_not_run_are_not_taken_for_computed(fake, call):
    ps = fake.ps
    plan, u = ps.ps_plan_create(ps.make_config(32, nu=1e-3)), np.zeros((3, 32, 32, 17), np.complex64).ctypes.data
    ens = ps.ps_ensemble_create([ps.make_config(32, nu=1e-3)])
    fake.fail(call, 1, ILLEGAL_ADDRESS)
    with pytest.raises(ps.PsError):
        ps.ps_rk_steps(plan, u, 1e-3, 0.0, 2)
    fake.fail(call, 1, ILLEGAL_ADDRESS)
    with pytest.raises(ps.PsError):
        ps.ps_ensemble_rk_steps(ens, [u], 1e-3, 0.0, 2, ps.ENS_GRAPH)
    fake.lib.fake_reset()
    ps.ps_rk_step(plan, u, 1e-3)
    ps.ps_ensemble_rk_steps(ens, [u], 1e-3, 0.0, 1, ps.ENS_SEQUENTIAL)
    assert _tables(fake) == 2
    ps.ps_ensemble_destroy(ens)
    ps.ps_plan_destroy(plan)
