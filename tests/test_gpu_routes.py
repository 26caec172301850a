"""The routes that a rule on sizes chooses: 512-point FP32 column lines (pairs of
threads), field-split z-inverse launches of small grids, one-line-at-a-time x
passes (MHD, Boussinesq, FP64), the pruned transforms of the training samples
and the closure's fields in the step's passes, at the lengths where each begins
and ends."""

import math

import numpy as np
import pytest

import oracle
from oracle import les as oles
from paper_1808_01309_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ps():
    import __graft_entry__
    __graft_entry__.build()
    from paper_1808_01309_gb300 import ps as _ps
    return _ps


def _dev(a, dtype=torch.complex64):
    return torch.from_numpy(np.ascontiguousarray(a)).to("cuda", dtype)


def _rel(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


@pytest.mark.parametrize("n", [(16, 512, 8), (8, 16, 512), (48, 512, 512), (512, 512, 8)], ids=str)
def test_512_point_lines(ps, n):
    """FP32 right-hand side, 2e-6 of the oracle as for every other length."""
    u = inputs.random_solenoidal_field(*n, seed=21, kmax=n)
    got = ps.Plan(*n, prec=ps.Precision.FP32, nu=1e-3).rhs(_dev(u)).cpu().numpy()
    assert _rel(got, oracle.rhs(u, oracle.Config(*n, nu=1e-3))) < 2e-6


def _state(eq, n):
    u = inputs.random_solenoidal_field(*n, seed=22, kmax=n)
    if eq == "MHD":
        return np.concatenate([u, inputs.random_solenoidal_field(*n, seed=23, kmax=n)])
    if eq == "BOUSSINESQ":
        return np.concatenate([u, inputs.random_scalar_field(*n, seed=24)])
    return u


@pytest.mark.parametrize("nx", [8, 16, 32, 48, 64, 96, 128, 192, 256, 512, 1024])
@pytest.mark.parametrize("eq", ["MHD", "BOUSSINESQ"])
def test_multi_field_rows(ps, eq, nx):
    """FP32 against FP64.  The curl of the FP32 u x B amplifies its rounding by
    |k|: 2e-6 up to |k| = 10, proportionally more above."""
    n = (nx, 16, 8)
    s = _state(eq, n)
    kw = dict(eq=getattr(ps.Equations, eq), nu=1e-3, eta=1e-3, kappa=1e-3, n_bv=1.5)
    ref = ps.Plan(*n, prec=ps.Precision.FP64, **kw).rhs(_dev(s, torch.complex128)).cpu().numpy()
    got = ps.Plan(*n, prec=ps.Precision.FP32, **kw).rhs(_dev(s)).cpu().numpy()
    amp = max(1.0, nx / 3.0 / 10.0) if eq == "MHD" else 1.0
    assert _rel(got, ref) < 2e-6 * amp


@pytest.mark.parametrize("n", [(16, 16, 16), (32, 8, 128), (128, 96, 64), (256, 64, 192)], ids=str)
@pytest.mark.parametrize("eq", ["HD", "MHD", "BOUSSINESQ"])
@pytest.mark.parametrize("prec", ["FP32", "FP64"])
def test_step_energy(ps, prec, eq, n):
    """The energy partials of split and whole z-inverse launches: the energy of
    the state a step starts from, summed in 64 bits."""
    dtype = torch.complex64 if prec == "FP32" else torch.complex128
    d = _dev(_state(eq, n), dtype)
    keep = oracle.dealias_mask(oracle.Config(*n))
    x = d.cpu().numpy().astype(np.complex128) * keep
    w = np.full(n[0] // 2 + 1, 2.0)
    w[0] = 1.0
    want = 0.5 * np.sum(w * np.abs(x) ** 2)
    plan = ps.Plan(*n, prec=getattr(ps.Precision, prec), eq=getattr(ps.Equations, eq), nu=1e-3, eta=1e-3, kappa=1e-3,
                   n_bv=1.0)
    plan.rk_step(d, 1e-4)
    assert abs(ps.ps_step_stats(plan.handle)[0] - want) < (1e-6 if prec == "FP32" else 1e-13) * want


@pytest.mark.parametrize("case", [(16, 16, 5), (48, 32, 10), (192, 16, 3), (256, 48, 15), (512, 64, 21)],
                         ids=lambda c: f"{c[0]}to{c[1]}kc{c[2]}")
def test_training_sample_stress(ps, case):
    """T against 64-bit transforms on the GPU; FP32 products of four transforms
    are good to 1e-5 of the mean square velocity."""
    nd, nl, kc = case
    gen = torch.Generator(device="cuda")
    gen.manual_seed(3)
    u = torch.fft.rfftn(torch.randn((3, nd, nd, nd), generator=gen, device="cuda"), dim=(-3, -2, -1), norm="forward")
    P = nl ** 3
    X, A, T = (torch.empty((P, k), device="cuda") for k in (5, 9, 6))
    ps.ps_les_training_sample(nd, u.contiguous(), nl, kc, None, X, A, T)
    i = torch.cat([torch.arange(kc + 1), torch.arange(-kc, 0)]).cuda()

    def box(f):
        o = torch.zeros((nl, nl, nl // 2 + 1), device="cuda", dtype=torch.complex128)
        o[(i % nl)[:, None], (i % nl)[None], :kc + 1] = f[(i % f.shape[0])[:, None], (i % f.shape[0])[None], :kc + 1]
        return o

    def inv(f, n):
        return torch.fft.irfftn(f, s=(n, n, n), norm="forward")

    v = [inv(u[c].to(torch.complex128), nd) for c in range(3)]
    b = [inv(box(u[c].to(torch.complex128)), nl) for c in range(3)]
    scale = float(sum((x * x).mean() for x in v))
    for m, (p, q) in enumerate(((0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2))):
        f = box(torch.fft.rfftn(v[p] * v[q], norm="forward")) - box(torch.fft.rfftn(b[p] * b[q], norm="forward"))
        err = (T[:, m].double() - inv(f, nl).reshape(-1)).abs().max()
        assert float(err) < 1e-5 * scale, m


@pytest.mark.parametrize("n", [(96, 16, 48), (128, 32, 16), (16, 192, 64), (256, 16, 32), (32, 16, 512)], ids=str)
def test_closure_fields_in_the_passes(ps, n):
    """The closure's right-hand side on lines of every length (the tolerance of
    the cubic cases)."""
    from paper_1808_01309_gb300 import les
    u = inputs.random_solenoidal_field(*n, seed=25, kmax=n)
    cfg = oracle.Config(*n, nu=5e-3)
    v = les.init_params(seed=4, out_scale=0.5)
    p, o = [], 0
    for _, shape in les.SHAPES:
        p.append(v[o:o + math.prod(shape)].reshape(shape).astype(np.float64))
        o += math.prod(shape)
    A = oles.gradient(u, cfg)
    lam = oles.invariants(A).reshape(5, -1)
    norm = dict(mean=lam.mean(1), std=lam.std(1), s_tau=0.05, s_A=math.sqrt(np.mean(np.sum(A * A, axis=(0, 1)))))
    keys = [name for name, _ in les.SHAPES]
    params = dict(zip(keys, p))
    plan = ps.Plan(*n, prec=ps.Precision.FP32, nu=5e-3)
    plan.set_closure(torch.from_numpy(v).cuda(), norm)
    got = plan.rhs(_dev(u)).cpu().numpy()
    ref = oles.les_rhs(u, cfg, params, norm, rnd=oles.bf16_round)
    assert _rel(got, ref) < 2e-4
