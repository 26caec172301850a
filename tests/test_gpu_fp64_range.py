"""The range that include/ps.h states for FP64 transforms: the advection of a
scalar of order one, u . grad theta, is linear in u, so a velocity 2^k times as
large gives 2^k times the tendency while its lines stay above 2^-937, and is off
by absolute errors near 2^-1021 below.

Tolerance: FP64 arithmetic rounds at 2^-53 wherever the exponents lie, about 30
times from the state to the tendency (transforms, products, transforms): 2^-48,
and 2^-45 holds it.  Below the range the absolute error of a mode is that of the
lines it comes from, times the gradient of theta (below 2^3) and the square root
of the lines' lengths (below 2^9) in all: 2^-1009 a mode, 2^-1002 in the norm of
at most 2^14 modes."""

import numpy as np
import pytest

from paper_1808_01309_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ps():
    import __graft_entry__
    __graft_entry__.build()
    from paper_1808_01309_gb300 import ps as _ps
    return _ps


@pytest.mark.parametrize("n", [(16, 16, 16), (48, 64, 8), (8, 512, 8), (512, 8, 16)], ids=str)
@pytest.mark.parametrize("k", [-600, -900, -980])
def test_advection_by_a_tiny_velocity(ps, k, n):
    u = inputs.random_solenoidal_field(*n, seed=31, kmax=n)
    th = inputs.random_scalar_field(*n, seed=32)
    plan = ps.Plan(*n, prec=ps.Precision.FP64, eq=ps.Equations.BOUSSINESQ, nu=0.0, kappa=0.0, n_bv=0.0)

    def tendency(scale):
        s = np.concatenate([np.ldexp(u.real, scale) + 1j * np.ldexp(u.imag, scale), th])
        return plan.rhs(torch.from_numpy(s).cuda()).cpu().numpy()[3]

    one, tiny = tendency(0), tendency(k)
    back = np.ldexp(tiny.real, -k) + 1j * np.ldexp(tiny.imag, -k)
    assert np.linalg.norm(back - one) <= 2.0 ** -45 * np.linalg.norm(one) + 2.0 ** (-1002 - k)
