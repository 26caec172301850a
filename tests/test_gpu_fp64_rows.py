"""FP64 MHD and Boussinesq right-hand sides against the oracle at row lengths that
the parity cases leave out, each with its own schedule, registers and rows per
CTA of the x pass: 1e-12, as for every FP64 right-hand side."""

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


@pytest.mark.parametrize("nx", [8, 48, 96, 128, 192, 256, 512, 1024])
@pytest.mark.parametrize("eq", ["MHD", "BOUSSINESQ"])
def test_rows_match_the_oracle(ps, eq, nx):
    n = (nx, 16, 8)
    u = inputs.random_solenoidal_field(*n, seed=41, kmax=n)
    second = inputs.random_solenoidal_field(*n, seed=42, kmax=n) if eq == "MHD" else inputs.random_scalar_field(*n, seed=43)
    s = np.concatenate([u, second])
    kw = dict(nu=1e-3, eta=2e-3) if eq == "MHD" else dict(nu=1e-3, kappa=2e-3, n_bv=1.5)
    rhs = oracle.mhd_rhs if eq == "MHD" else oracle.boussinesq_rhs
    ref = rhs(s, oracle.Config(*n, **kw))
    plan = ps.Plan(*n, prec=ps.Precision.FP64, eq=getattr(ps.Equations, eq), **kw)
    got = plan.rhs(torch.from_numpy(s).cuda()).cpu().numpy()
    assert np.linalg.norm(got - ref) <= 1e-12 * np.linalg.norm(ref)
