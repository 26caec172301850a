"""The FP64 passes' block fixed-point transforms (csrc/ps_fix.cuh): accuracy at
every line length, exact equivariance under powers of two, zero lines and
non-finite values.

Tolerance of the accuracy test: a right-hand side passes six transforms of at
most four stages; each stage rounds at q = 2^-62 L1 <= 2^-61 (L1 <= N rms, so
q <= 2^-51 rms at 1024 points), which with the FP64 pointwise work and the
oracle's own transforms (about 10 roundings of 2^-53 each) stays below 50 x
2^-52 = 1.1e-14 of the field."""

import math

import numpy as np
import pytest

import oracle
from paper_1808_01309_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ps():
    import __graft_entry__
    __graft_entry__.build()
    from paper_1808_01309_gb300 import ps as _ps
    return _ps


def _rhs(ps, n, u, **kw):
    plan = ps.Plan(*n, prec=ps.Precision.FP64, **kw)
    out = plan.rhs(torch.from_numpy(np.ascontiguousarray(u)).cuda())
    torch.cuda.synchronize()
    return out


@pytest.mark.parametrize("n", [(8, 16, 32), (48, 64, 96), (192, 8, 128), (256, 48, 8), (16, 512, 8), (512, 8, 192),
                               (8, 256, 1024), (1024, 16, 8)], ids=str)
def test_accuracy(ps, n):
    u = inputs.random_solenoidal_field(*n, seed=5, kmax=n)
    ref = oracle.rhs(u, oracle.Config(*n, nu=1e-3))
    got = _rhs(ps, n, u, nu=1e-3).cpu().numpy()
    assert np.linalg.norm(got - ref) <= 1.1e-14 * np.linalg.norm(ref)


@pytest.mark.parametrize("k", [-400, -60, 1, 33, 300])
def test_powers_of_two_scale_exactly(ps, k):
    """Without diffusion the right-hand side is quadratic, and neither FP64 nor
    the block scaling rounds differently after a change of exponents."""
    n = (48, 32, 16)
    u = inputs.random_solenoidal_field(*n, seed=6, kmax=n)
    one, two = _rhs(ps, n, u, nu=0.0), _rhs(ps, n, u * 2.0 ** k, nu=0.0)
    assert torch.equal(two, one * 2.0 ** (2 * k))


def test_zero_state(ps):
    n = (32, 32, 32)
    assert not _rhs(ps, n, np.zeros((3, 32, 32, 17), complex), nu=1e-3).any()


@pytest.mark.parametrize("bad", [math.nan, math.inf, -math.inf])
def test_non_finite_values_reach_every_retained_mode(ps, bad):
    n = (32, 64, 16)
    u = inputs.random_solenoidal_field(*n, seed=7, kmax=n)
    u[1, 3, 2, 4] = bad
    got = _rhs(ps, n, u, nu=1e-3).cpu().numpy()
    kx, ky, kz = (-(-m // 3) - 1 for m in n)
    q, r = np.fft.fftfreq(n[1], 1 / n[1]), np.fft.fftfreq(n[2], 1 / n[2])
    keep = (abs(r) <= kz)[:, None, None] & (abs(q) <= ky)[None, :, None] & (np.arange(n[0] // 2 + 1) <= kx)
    keep[0, 0, 0] = False
    assert np.isnan(got[:, keep]).all()
