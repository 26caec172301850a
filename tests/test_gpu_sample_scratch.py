"""The scratch block that ps_les_training_sample keeps between calls: the same
outputs from a kept block, from concurrent calls on several streams and after a
change of size, and the memory back once a plan is destroyed."""

import threading

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ps():
    import __graft_entry__
    __graft_entry__.build()
    from paper_1808_01309_gb300 import ps as _ps
    return _ps


def _input(n, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    x = torch.randn((3, n, n, n), generator=gen, device="cuda")
    return torch.fft.rfftn(x, dim=(-3, -2, -1), norm="forward").contiguous()


def _sample(ps, u, n, nl, kc, stream=None):
    out = [torch.empty((nl ** 3, k), device="cuda") for k in (5, 9, 6)]
    ps.ps_les_training_sample(n, u, nl, kc, None, *out, **({} if stream is None else dict(stream=stream)))
    torch.cuda.synchronize()
    return out


def _same(a, b):
    return all(torch.equal(x, y) for x, y in zip(a, b))


def test_kept_block_and_sizes(ps):
    big, small = _input(128, 1), _input(32, 2)
    first, tiny = _sample(ps, big, 128, 32, 8), _sample(ps, small, 32, 16, 5)
    for _ in range(2):
        assert _same(_sample(ps, big, 128, 32, 8), first)
        assert _same(_sample(ps, small, 32, 16, 5), tiny)


def test_concurrent_calls(ps):
    u = [_input(64, 10 + i) for i in range(4)]
    ref = [_sample(ps, x, 64, 32, 10) for x in u]
    ok = [False] * 4

    def work(i):
        s = torch.cuda.Stream()
        ok[i] = all(_same(_sample(ps, u[i], 64, 32, 10, s.cuda_stream), ref[i]) for _ in range(10))

    threads = [threading.Thread(target=work, args=(i,)) for i in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert all(ok)


def test_memory_is_given_back(ps):
    u = _input(256, 3)
    plan = ps.Plan(16, prec=ps.Precision.FP32, nu=1e-3)
    _sample(ps, u, 256, 64, 21)
    kept = torch.cuda.mem_get_info()[0]
    plan.close()
    assert torch.cuda.mem_get_info()[0] - kept > 200 << 20
