"""The calls this library is timed on, as its users make them.

Each case is one public entry point on seeded synthetic inputs, made on the
GPU.  Grids, viscosities, time steps and options are those of
paper_1808_01309_gb300/workloads.py, of the tests and of bench.py; the fields
are solenoidal with a developed-turbulence spectrum over the whole retained
set, so that every mode carries a value.

  kind "step"      one Runge-Kutta step (ps_rk_step), in place on the state
  kind "steps"     several steps replayed as one graph (ps_rk_steps)
  kind "rhs"       one right-hand side (ps_rhs)
  kind "ensemble"  steps of many independent members (ps_ensemble_rk_steps)
  kind "les"       graph-replayed LES steps with the learned closure attached
  kind "train"     one full-batch iteration of the closure's stress fit
                   (ps_mlp_grad_tb, ps_mlp_adam)
  kind "sample"    training pairs of one DNS snapshot (ps_les_training_sample)
  kind "diag"      the diagnostics of a state (ps_diagnostics)
"""

from __future__ import annotations

import math

import numpy as np
import torch

from paper_1808_01309_gb300 import inputs, les, ps, workloads

DEV = "cuda"
TWO_PI = 2.0 * math.pi
PREC = {"fp32": ps.Precision.FP32, "fp64": ps.Precision.FP64}
EQ = {"hd": ps.Equations.HD, "mhd": ps.Equations.MHD, "boussinesq": ps.Equations.BOUSSINESQ}
DEALIAS = {"cubic": ps.Dealias.CUBIC, "spherical": ps.Dealias.SPHERICAL, "none": ps.Dealias.NONE}
NCOMP = {"hd": 3, "mhd": 6, "boussinesq": 4}
# order of the symmetric stress components
SYM = ((0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2))


def _solve(kind, name=None, nx=64, ny=None, nz=None, prec="fp32", eq="hd", dealias="cubic", order=4, nu=2e-3,
           dt=1e-3, nsteps=1, forced=True, lz=TWO_PI):
    c = dict(kind=kind, nx=nx, ny=ny or nx, nz=nz or nx, prec=prec, eq=eq, dealias=dealias, order=order, nu=nu, dt=dt,
             nsteps=nsteps, forced=forced, lz=lz)
    return dict(name=name, **c) if name else c


def listed():
    return [
        # the smallest solve, in the paper's precision: a verification run, bound by launches
        _solve("step", "hd_32_fp64_rk2", 32, prec="fp64", order=2, nu=1e-2, forced=False),
        # a small DNS (or an LES without a closure) advanced as a user loops over it
        _solve("steps", "hd_64_graph10", 64, nu=5e-3, nsteps=10),
        # a bare right-hand side, for users with a time integrator of their own
        _solve("rhs", "hd_192_spherical_rhs", 192, dealias="spherical"),
        # the ordinary DNS step
        _solve("step", "hd_256", 256),
        # the headline DNS step
        _solve("step", "hd_512", 512),
        # the same solver in double precision (the paper's precision)
        _solve("step", "hd_256_fp64", 256, prec="fp64"),
        # magnetohydrodynamics: twice the fields per pass
        _solve("step", "mhd_256", 256, eq="mhd"),
        # stratified flow in a flat box on an anisotropic grid
        _solve("step", "boussinesq_512x512x128", 512, 512, 128, eq="boussinesq", lz=TWO_PI / 4),
        # a parameter study: 48 independent members of three sizes
        dict(name="ensemble_48", kind="ensemble", sizes=",".join(str(n) for n in workloads.ENSEMBLE_SIZES), nsteps=2,
             dt=1e-3),
        # a large-eddy simulation with the learned closure
        dict(name="les_64_graph10", kind="les", n=64, nsteps=10, dt=5e-3, nu=2e-3),
        # one iteration of the closure's fit on eight 64^3 snapshots
        dict(name="train_2m", kind="train", count=8 * 64 ** 3),
        # training pairs of a 64^3 LES from one 256^3 snapshot
        dict(name="sample_256_64", kind="sample", n_dns=256, n_les=64, kc=21),
    ]


SIZES = (16, 32, 48, 64, 96, 128, 192, 256, 512)
LES_SIZES = (32, 48, 64, 96, 128)


def draw(rng):
    """One more case of the listed kinds: every grid length, precision,
    equation set, truncation, order and forcing, and ragged sample counts."""
    kind = rng.choice(("step", "step", "step", "step", "steps", "rhs", "ensemble", "les", "train", "sample", "diag"))
    if kind in ("step", "steps", "rhs", "diag"):
        eq = rng.choice(("hd", "hd", "mhd", "boussinesq"))
        prec = rng.choice(("fp32", "fp32", "fp64"))
        weight = {"hd": 1.0, "mhd": 2.0, "boussinesq": 1.5}[eq] * (8.0 if prec == "fp64" else 1.0)
        cap = 128 ** 3 if kind == "steps" else 512 ** 3 / weight
        while True:
            base = rng.choice(SIZES)
            n = [base] + [rng.choice((base, base, rng.choice(SIZES))) for _ in range(2)]
            rng.shuffle(n)
            if 2 ** 15 <= n[0] * n[1] * n[2] <= cap:
                break
        return _solve(kind, None, n[0], n[1], n[2], prec=prec, eq=eq,
                      dealias=rng.choice(("cubic", "cubic", "spherical", "none")), order=rng.choice((2, 4, 4)),
                      nu=5e-3, dt=1e-3, nsteps=rng.choice((3, 7, 10)) if kind == "steps" else 1,
                      forced=rng.random() < 0.6, lz=rng.choice((TWO_PI, TWO_PI / 2, 3.0)))
    if kind == "ensemble":
        sizes = [rng.choice((32, 48, 64, 96, 128)) for _ in range(rng.randint(2, 24))]
        return dict(kind=kind, sizes=",".join(str(n) for n in sizes), nsteps=rng.choice((1, 2, 3)), dt=1e-3)
    if kind == "les":
        return dict(kind=kind, n=rng.choice(LES_SIZES), nsteps=rng.choice((2, 5, 10)), dt=2e-3, nu=2e-3)
    if kind == "train":
        return dict(kind=kind, count=int(math.exp(rng.uniform(math.log(2 ** 10), math.log(2 ** 22)))))
    n_les = rng.choice((32, 48, 64, 96))
    n_dns = rng.choice([n for n in (64, 96, 128, 192, 256) if n >= n_les])
    return dict(kind="sample", n_dns=n_dns, n_les=n_les, kc=rng.randint(max(2, n_les // 8), -(-n_les // 3) - 1))


# ---- fields -------------------------------------------------------------------

class _Grid:
    """Wavenumbers, retained set and Hermitian weight of a case, in 64 bits."""

    def __init__(self, nx, ny, nz, lz=TWO_PI, dealias="cubic"):
        self.n = (nz, ny, nx)
        self.box = (TWO_PI, TWO_PI, lz)
        p = torch.arange(nx // 2 + 1, device=DEV, dtype=torch.int64).view(1, 1, -1)
        q = (torch.fft.fftfreq(ny, 1.0 / ny, device=DEV, dtype=torch.float64).round().long()).view(1, -1, 1)
        r = (torch.fft.fftfreq(nz, 1.0 / nz, device=DEV, dtype=torch.float64).round().long()).view(-1, 1, 1)
        half = [n // 2 - 1 if dealias == "none" else -(-n // 3) - 1 for n in (nx, ny, nz)]
        self.half = half
        self.keep = (p <= half[0]) & (q.abs() <= half[1]) & (r.abs() <= half[2])
        if dealias == "spherical":
            self.keep = self.keep & ((3.0 * p / nx) ** 2 + (3.0 * q / ny) ** 2 + (3.0 * r / nz) ** 2 < 1.0)
        self.k = (TWO_PI / self.box[0] * p.double(), TWO_PI / self.box[1] * q.double(),
                  TWO_PI / self.box[2] * r.double())
        self.k2 = self.k[0] ** 2 + self.k[1] ** 2 + self.k[2] ** 2
        self.w = torch.full((nx // 2 + 1,), 2.0, device=DEV, dtype=torch.float64)
        self.w[0] = 1.0

    def inverse(self, f):
        return torch.fft.irfftn(f, s=self.n, dim=(-3, -2, -1), norm="forward")

    def forward(self, f):
        return torch.fft.rfftn(f, dim=(-3, -2, -1), norm="forward")

    def project(self, v):
        s = (self.k[0] * v[0] + self.k[1] * v[1] + self.k[2] * v[2]) / self.k2.clamp(min=1e-300)
        for c in range(3):
            v[c] -= self.k[c] * s
        return v


def _hermitian(f):
    """Exact Hermitian symmetry of the kx = 0 plane."""
    plane = f[..., 0]
    mirror = torch.roll(torch.flip(plane, (-2, -1)), (1, 1), (-2, -1))
    f[..., 0] = 0.5 * (plane + mirror.conj())
    return f


def _random(g, ncomp, gen, dtype, solenoidal=True):
    """Random retained modes, E(K) ~ K^4 at small and K^-5/3 at large K with an
    exponential tail, half the sum of w |f|^2 equal to 0.5."""
    real = torch.float32 if dtype == torch.complex64 else torch.float64
    f = torch.empty((ncomp,) + g.n[:2] + (g.n[2] // 2 + 1,), device=DEV, dtype=dtype)
    k = torch.sqrt(g.k2)
    kmax = min(h * TWO_PI / b for h, b in zip(g.half, g.box))
    amp = k / (1.0 + (k / 3.0) ** 2) ** (17.0 / 12.0) * torch.exp(-1.5 * k / kmax) * g.keep
    amp[0, 0, 0] = 0.0
    for c in range(ncomp):
        f[c] = torch.fft.rfftn(torch.randn(g.n, generator=gen, device=DEV, dtype=real), norm="ortho")
        f[c] *= amp.to(real)
    if solenoidal:
        k2 = g.k2.to(real).clamp(min=1e-30)
        s = (g.k[0].to(real) * f[0] + g.k[1].to(real) * f[1] + g.k[2].to(real) * f[2]) / k2
        for c in range(3):
            f[c] -= g.k[c].to(real) * s
        del s
    _hermitian(f)
    e = sum(float((0.5 * g.w * (f[c].real.double() ** 2 + f[c].imag.double() ** 2)).sum()) for c in range(ncomp))
    f *= math.sqrt(0.5 / e)
    return f


def _forcing(g, gen, dtype):
    """Constant solenoidal forcing on 2 <= |k| <= 3, rms 0.25."""
    f = _random(g, 3, gen, torch.complex128)
    f *= ((g.k2 >= 4.0 - 1e-9) & (g.k2 <= 9.0 + 1e-9))
    ms = float(sum((g.w * f[c].abs() ** 2).sum() for c in range(3)))
    return (f * (0.25 / math.sqrt(ms) if ms > 0 else 0.0)).to(dtype).contiguous()


def _gen(seed):
    gen = torch.Generator(device=DEV)
    gen.manual_seed(1 + int(seed))
    return gen


def _solve_inputs(c, seed):
    g = _Grid(c["nx"], c["ny"], c["nz"], c["lz"], c["dealias"])
    gen = _gen(seed)
    dtype = torch.complex64 if c["prec"] == "fp32" else torch.complex128
    u = _random(g, 3, gen, dtype)
    if c["eq"] == "mhd":
        u = torch.cat([u, _random(g, 3, gen, dtype)])
    elif c["eq"] == "boussinesq":
        u = torch.cat([u, _random(g, 1, gen, dtype, solenoidal=False)])
    f = _forcing(g, gen, dtype) if c["forced"] else None
    return g, u.contiguous(), f


# ---- the closure's data ---------------------------------------------------------

def _mm(X, Y):
    """Products of [..., 3, 3] matrices, elementwise (batched 3 x 3 GEMMs are slow)."""
    return (X.unsqueeze(-1) * Y.unsqueeze(-3)).sum(-2)


def _invariants(A):
    """tr S^2, tr R^2, tr S^3, tr S R^2, tr S^2 R^2 of A[..., 3, 3]."""
    S, R = 0.5 * (A + A.mT), 0.5 * (A - A.mT)
    S2, R2 = _mm(S, S), _mm(R, R)
    return torch.stack([(S * S.mT).sum((-2, -1)), (R * R.mT).sum((-2, -1)), (S2 * S.mT).sum((-2, -1)),
                        (S * R2.mT).sum((-2, -1)), (S2 * R2.mT).sum((-2, -1))], -1)


def _basis(A, s_A):
    """The six basis tensors of A/s_A as [..., 6 tensors, 6 components]."""
    S, R = 0.5 * (A + A.mT) / s_A, 0.5 * (A - A.mT) / s_A
    S2, R2 = _mm(S, S), _mm(R, R)
    eye = torch.eye(3, device=A.device, dtype=A.dtype)
    SR2 = _mm(S, R2)

    def tr(X):
        return X.diagonal(dim1=-2, dim2=-1).sum(-1)[..., None, None]

    T = (S, _mm(S, R) - _mm(R, S), S2 - tr(S2) * eye / 3, R2 - tr(R2) * eye / 3, _mm(R, S2) - _mm(S2, R),
         _mm(R2, S) + SR2 - 2.0 * tr(SR2) * eye / 3)
    return torch.stack([torch.stack([t[..., i, j] for i, j in SYM], -1) for t in T], -2)


def _network(params, X):
    out, o = [], 0
    for _, shape in les.SHAPES:
        n = math.prod(shape)
        out.append(params[o:o + n].view(shape))
        o += n
    W1, b1, W2, b2, W3, b3 = out

    def gelu(x):
        return torch.nn.functional.gelu(x, approximate="tanh")

    return gelu(gelu(X @ W1 + b1) @ W2 + b2) @ W3 + b3


def _gradients(count, gen):
    """Velocity gradients of a turbulent flow: traceless, with heavy tails."""
    A = torch.randn((count, 3, 3), generator=gen, device=DEV, dtype=torch.float32)
    A -= A.diagonal(dim1=-2, dim2=-1).sum(-1)[:, None, None] * torch.eye(3, device=DEV) / 3
    A *= torch.exp(0.4 * torch.randn((count, 1, 1), generator=gen, device=DEV, dtype=torch.float32))
    return A.contiguous()


def _norm_of(A, s_tau):
    lam = _invariants(A.double())
    s_A = math.sqrt(float((A.double() ** 2).sum((-2, -1)).mean()))
    return [float(x) for x in lam.mean(0)] + [float(x) for x in lam.std(0)] + [s_tau, s_A]


def _params(seed):
    return torch.from_numpy(les.init_params(seed=int(seed) % (2 ** 31), out_scale=0.1)).to(DEV)


def _grad_field(g, u):
    A = torch.stack([torch.stack([g.inverse(1j * g.k[j] * u[i]) for j in range(3)]) for i in range(3)])
    return A.permute(2, 3, 4, 0, 1).contiguous()


def _les_inputs(c, seed):
    g = _Grid(c["n"], c["n"], c["n"])
    gen = _gen(seed)
    u = _random(g, 3, gen, torch.complex64)
    f = _forcing(g, gen, torch.complex64)
    norm = _norm_of(_grad_field(g, u.to(torch.complex128)).view(-1, 3, 3), 0.02)
    return g, u, f, _params(seed), norm


def _train_inputs(c, seed):
    gen = _gen(seed)
    A = _gradients(c["count"], gen)
    norm = _norm_of(_gradients(1 << 16, gen), 0.02)
    mean, std = (torch.tensor(v, device=DEV, dtype=torch.float32) for v in (norm[:5], norm[5:10]))
    X = ((_invariants(A) - mean) / std).contiguous()
    S = 0.5 * (A + A.mT) / norm[11]
    T = torch.stack([-0.3 * S[:, i, j] for i, j in SYM], -1)
    T = norm[10] * (T + torch.randn(T.shape, generator=gen, device=DEV, dtype=torch.float32))
    # a fit some way on: parameters and moments of a previous iteration
    m = 1e-4 * torch.randn(ps.MLP_NPARAM, generator=gen, device=DEV, dtype=torch.float32)
    v = 1e-6 * (1.0 + torch.rand(ps.MLP_NPARAM, generator=gen, device=DEV, dtype=torch.float32))
    return dict(X=X, A=A.view(-1, 9), T=T.contiguous(), params=_params(seed), m=m, v=v, s_tau=norm[10], s_A=norm[11],
                step=1000)


def _sample_inputs(c, seed):
    g = _Grid(c["n_dns"], c["n_dns"], c["n_dns"])
    gen = _gen(seed)
    u = _random(g, 3, gen, torch.complex64)
    return g, u, _norm_of(_gradients(1 << 14, gen), 1.0)


class _Ensemble:
    """One ps_ensemble, destroyed with the object."""

    def __init__(self, cfgs):
        self.handle = ps.ps_ensemble_create(cfgs)

    def __del__(self):
        if ps is not None and ps.load is not None:
            ps.load().ps_ensemble_destroy(self.handle)


def _members(c, seed):
    out = []
    for i, n in enumerate(int(x) for x in c["sizes"].split(",")):
        out.append((_Grid(n, n, n), _random(_Grid(n, n, n), 3, _gen(1000 * int(seed) + i), torch.complex64),
                    inputs.ensemble_viscosity(i)))
    return out


# ---- the calls --------------------------------------------------------------------

def prepare(case, seed):
    c, kind = case, case["kind"]
    if kind in ("step", "steps", "rhs", "diag"):
        _, u, f = _solve_inputs(c, seed)
        plan = ps.Plan(c["nx"], c["ny"], c["nz"], lz=c["lz"], prec=PREC[c["prec"]], eq=EQ[c["eq"]],
                       dealias=DEALIAS[c["dealias"]], rk_order=c["order"], nu=c["nu"], eta=c["nu"],
                       kappa=c["nu"], n_bv=1.0, forcing=f)
        s = dict(kind=kind, plan=plan, u=u, dt=c["dt"], nsteps=c["nsteps"])
        if kind == "rhs":
            s["out"] = torch.empty_like(u)
        return s
    if kind == "ensemble":
        mem = _members(c, seed)
        ens = _Ensemble([ps.make_config(g.n[2], nu=nu, rk_order=4) for g, _, nu in mem])
        return dict(kind=kind, ens=ens, states=[u for _, u, _ in mem], dt=c["dt"], nsteps=c["nsteps"])
    if kind == "les":
        _, u, f, params, norm = _les_inputs(c, seed)
        plan = ps.Plan(c["n"], prec=ps.Precision.FP32, nu=c["nu"], rk_order=4, forcing=f)
        plan.set_closure(params, norm)
        return dict(kind=kind, plan=plan, u=u, dt=c["dt"], nsteps=c["nsteps"])
    if kind == "train":
        s = _train_inputs(c, seed)
        return dict(kind=kind, grad=torch.empty_like(s["params"]),
                    loss=torch.empty(1, device=DEV, dtype=torch.float64), **s)
    g, u, norm = _sample_inputs(c, seed)
    n = c["n_les"] ** 3
    buf = [torch.empty((n, k), device=DEV, dtype=torch.float32) for k in (5, 9, 6)]
    return dict(kind=kind, u=u, norm=norm, n_dns=c["n_dns"], n_les=c["n_les"], kc=c["kc"], buf=buf)


def run(state):
    s, kind = state, state["kind"]
    if kind == "step":
        return s["plan"].rk_step(s["u"], s["dt"])
    if kind in ("steps", "les"):
        return s["plan"].rk_steps(s["u"], s["dt"], s["nsteps"])
    if kind == "rhs":
        return s["plan"].rhs(s["u"], out=s["out"])
    if kind == "diag":
        return _diag_output(s["plan"].diagnostics(s["u"]))
    if kind == "ensemble":
        ps.ps_ensemble_rk_steps(s["ens"].handle, s["states"], s["dt"], 0.0, s["nsteps"])
        return s["states"]
    if kind == "train":
        ps.ps_mlp_grad_tb(s["params"], s["X"], s["A"], s["T"], s["X"].shape[0], s["s_A"], s["s_tau"], s["grad"],
                          s["loss"])
        ps.ps_mlp_adam(s["params"], s["grad"], s["m"], s["v"], s["step"], 1e-3)
        s["step"] += 1
        return dict(params=s["params"], m=s["m"], v=s["v"], grad=s["grad"], loss=s["loss"])
    X, A, T = s["buf"]
    ps.ps_les_training_sample(s["n_dns"], s["u"], s["n_les"], s["kc"], s["norm"], X, A, T)
    return [X, A, T]


DIAG = ("energy", "enstrophy", "helicity", "max_u", "cfl_dt", "magnetic_energy", "cross_helicity", "magnetic_helicity",
        "potential_energy")


def _diag_output(d):
    return dict({k: d[k] for k in DIAG}, spectrum=np.array(d["spectrum"]))


# ---- the work a call cannot do without -----------------------------------------------

def _rhs_flops(n, fields_in, fields_out):
    return (fields_in + fields_out) * 2.5 * n * math.log2(n) + 40.0 * n


def work(case):
    c, kind = case, case["kind"]
    if kind in ("step", "steps", "rhs", "diag"):
        n = c["nx"] * c["ny"] * c["nz"]
        state = NCOMP[c["eq"]] * c["nz"] * c["ny"] * (c["nx"] // 2 + 1) * (8 if c["prec"] == "fp32" else 16)
        fin, fout = {"hd": (6, 3), "mhd": (12, 6), "boussinesq": (9, 4)}[c["eq"]]
        evals = 1 if kind == "rhs" else c["order"] * c["nsteps"]
        if kind == "diag":
            return {"bytes": state, "flops": 3 * 2.5 * n * math.log2(n) + 20.0 * n}
        return {"bytes": 2 * state * (c["nsteps"] if kind == "steps" else 1), "flops": evals * _rhs_flops(n, fin, fout)}
    if kind == "ensemble":
        sizes = [int(x) for x in c["sizes"].split(",")]
        return {"bytes": c["nsteps"] * sum(2 * 3 * n * n * (n // 2 + 1) * 8 for n in sizes),
                "flops": c["nsteps"] * sum(4 * _rhs_flops(n ** 3, 6, 3) for n in sizes)}
    mlp = 2 * (5 * 64 + 64 * 64 + 64 * 6)
    if kind == "les":
        n = c["n"] ** 3
        return {"bytes": c["nsteps"] * 2 * 3 * c["n"] ** 2 * (c["n"] // 2 + 1) * 8,
                "flops": c["nsteps"] * 4 * (_rhs_flops(n, 6, 3) + 15 * 2.5 * n * math.log2(n) + (mlp + 800) * n)}
    if kind == "train":
        return {"bytes": c["count"] * 20 * 4 + 8 * ps.MLP_NPARAM * 4, "flops": c["count"] * (3 * mlp + 800)}
    nd, nl = c["n_dns"] ** 3, c["n_les"] ** 3
    return {"bytes": 3 * c["n_dns"] ** 2 * (c["n_dns"] // 2 + 1) * 8 + 20 * 4 * nl,
            "flops": 9 * 2.5 * nd * math.log2(nd) + 24 * 2.5 * nl * math.log2(nl)}


# ---- the same in 64 bits ----------------------------------------------------------------

def _curl(g, u):
    k = g.k
    return [1j * (k[1] * u[2] - k[2] * u[1]), 1j * (k[2] * u[0] - k[0] * u[2]), 1j * (k[0] * u[1] - k[1] * u[0])]


def _cross(a, b):
    return [a[1] * b[2] - a[2] * b[1], a[2] * b[0] - a[0] * b[2], a[0] * b[1] - a[1] * b[0]]


def _tendency(g, c, u, f, closure=None):
    """The right-hand side without the diffusive terms."""
    v = [g.inverse(u[i]) for i in range(3)]
    om = [g.inverse(x) for x in _curl(g, u)]
    n = _cross(v, om)
    del om
    out = torch.empty_like(u)
    if c["eq"] == "mhd":
        b = [g.inverse(u[3 + i]) for i in range(3)]
        j = [g.inverse(x) for x in _curl(g, u[3:])]
        n = [x + y for x, y in zip(n, _cross(j, b))]
        del j
        e = [g.forward(x) for x in _cross(v, b)]
        for i, x in enumerate(_curl(g, e)):
            out[3 + i] = x
    for i in range(3):
        out[i] = g.forward(n[i])
        if f is not None:
            out[i] += f[i]
        if closure is not None:
            out[i] += closure[i]
    if c["eq"] == "boussinesq":
        adv = sum(v[i] * g.inverse(1j * g.k[i] * u[3]) for i in range(3))
        out[2] -= u[3]
        out[3] = u[2] - g.forward(adv)
    out[:3] = g.project(out[:3])
    out[:3, 0, 0, 0] = 0.0
    return out * g.keep


def _exact_step(g, c, u, f, dt, order, nu, closure=None):
    def R(x):
        return _tendency(g, c, x, f, closure(x) if closure else None)

    E = torch.exp(-0.5 * nu * dt * g.k2)
    k1 = R(u)
    if order == 2:
        k2 = R(E * E * (u + dt * k1))
        return E * E * (u + 0.5 * dt * k1) + 0.5 * dt * k2
    acc = E * E * k1
    k2 = R(E * (u + 0.5 * dt * k1))
    acc += 2.0 * E * k2
    k3 = R(E * u + 0.5 * dt * k2)
    acc += 2.0 * E * k3
    acc += R(E * E * u + dt * E * k3)
    return E * E * u + dt / 6.0 * acc


def _exact_solve(c, seed):
    g, u, f = _solve_inputs(c, seed)
    u = u.to(torch.complex128)
    f = None if f is None else f.to(torch.complex128)
    if c["kind"] == "rhs":
        return _tendency(g, c, u, f) - c["nu"] * g.k2 * u
    if c["kind"] == "diag":
        return _exact_diag(g, c, u)
    for _ in range(c["nsteps"]):
        u = _exact_step(g, c, u, f, c["dt"], c["order"], c["nu"])
    return u


def _exact_diag(g, c, u):
    def total(x):
        return float((g.w * x).sum())

    def dot(a, b):
        return sum((x.conj() * y).real for x, y in zip(a, b))

    om = _curl(g, u)
    e = 0.5 * dot(u[:3], u[:3])
    shell = torch.floor(torch.sqrt(g.k2) + 0.5).long()
    top = math.floor(math.sqrt(sum((h * TWO_PI / b) ** 2 for h, b in zip(g.half, g.box))) + 0.5)
    spec = torch.zeros(int(shell.max()) + 1, device=DEV, dtype=torch.float64)
    spec.index_add_(0, shell.reshape(-1), (g.w * e).reshape(-1))
    max_u = math.sqrt(float(sum(g.inverse(u[i]) ** 2 for i in range(3)).max()))
    d = dict(energy=total(e), enstrophy=0.5 * total(dot(om, om)), helicity=total(dot(u[:3], om)), max_u=max_u,
             cfl_dt=0.5 * min(b / n for b, n in zip(g.box, reversed(g.n))) / max_u, magnetic_energy=0.0,
             cross_helicity=0.0, magnetic_helicity=0.0, potential_energy=0.0)
    if c["eq"] == "mhd":
        b, j = u[3:], _curl(g, u[3:])
        d.update(magnetic_energy=0.5 * total(dot(b, b)), cross_helicity=total(dot(u[:3], b)),
                 magnetic_helicity=total(dot(j, b) / g.k2.clamp(min=1e-300) * (g.k2 > 0)))
    if c["eq"] == "boussinesq":
        d["potential_energy"] = 0.5 * total(dot(u[3:], u[3:]))
    spec = spec.cpu().numpy()
    out = np.zeros(top + 1)
    out[:min(top + 1, spec.size)] = spec[:top + 1]
    return dict(d, spectrum=out)


def _exact_les(c, seed):
    g, u, f, params, norm = _les_inputs(c, seed)
    cc = dict(eq="hd")
    mean, std = (torch.tensor(v, device=DEV, dtype=torch.float64) for v in (norm[:5], norm[5:10]))
    pd = params.double()

    def closure(x):
        A = _grad_field(g, x)
        y = _network(pd, (_invariants(A) - mean) / std)
        tau = norm[10] * torch.einsum("...n,...nm->m...", y, _basis(A, norm[11]))
        th = [g.forward(tau[m]) for m in range(6)]
        idx = ((0, 3, 4), (3, 1, 5), (4, 5, 2))
        return [-1j * sum(g.k[j] * th[idx[i][j]] for j in range(3)) for i in range(3)]

    u, f = u.to(torch.complex128), f.to(torch.complex128)
    for _ in range(c["nsteps"]):
        u = _exact_step(g, cc, u, f, c["dt"], 4, c["nu"], closure)
    return u


def _exact_train(c, seed):
    s = _train_inputs(c, seed)
    p = s["params"].double().requires_grad_(True)
    n, loss = s["X"].shape[0], 0.0
    for i in range(0, n, 1 << 19):
        sl = slice(i, min(n, i + (1 << 19)))
        y = _network(p, s["X"][sl].double())
        B = _basis(s["A"][sl].double().view(-1, 3, 3), s["s_A"])
        e = torch.einsum("bn,bnm->bm", y, B) - s["T"][sl].double() / s["s_tau"]
        part = (e * e).sum() / (n * 6)
        part.backward()
        loss += float(part)
    with torch.no_grad():
        grad = p.grad
        m = 0.9 * s["m"].double() + 0.1 * grad
        v = 0.999 * s["v"].double() + 0.001 * grad ** 2
        q = p - 1e-3 * (m / (1 - 0.9 ** s["step"])) / (torch.sqrt(v / (1 - 0.999 ** s["step"])) + 1e-8)
    return dict(params=q.detach(), m=m, v=v, grad=grad, loss=torch.tensor([loss], device=DEV, dtype=torch.float64))


def _exact_sample(c, seed):
    g, u, norm = _sample_inputs(c, seed)
    u = u.to(torch.complex128)
    nl, nd, kc = c["n_les"], c["n_dns"], c["kc"]
    gl = _Grid(nl, nl, nl)

    def box(f):
        out = torch.zeros((nl, nl, nl // 2 + 1), device=DEV, dtype=torch.complex128)
        idx = torch.cat([torch.arange(kc + 1), torch.arange(-kc, 0)]).to(DEV)
        out[(idx % nl)[:, None], (idx % nl)[None], :kc + 1] = f[(idx % nd)[:, None], (idx % nd)[None], :kc + 1]
        return out

    v = [g.inverse(u[i]) for i in range(3)]
    ub = torch.stack([box(u[i]) for i in range(3)])
    vb = [gl.inverse(ub[i]) for i in range(3)]
    T = torch.stack([gl.inverse(box(g.forward(v[i] * v[j])) - _box_only(gl.forward(vb[i] * vb[j]), kc))
                     for i, j in SYM], -1)
    A = _grad_field(gl, ub)
    mean, std = (torch.tensor(x, device=DEV, dtype=torch.float64) for x in (norm[:5], norm[5:10]))
    X = (_invariants(A) - mean) / std
    return [X.reshape(-1, 5), A.reshape(-1, 9), T.reshape(-1, 6)]


def _box_only(f, kc):
    n = f.shape[0]
    i = torch.arange(n, device=DEV)
    s = torch.where(i < (n + 1) // 2, i, i - n).abs() <= kc
    return f * s[:, None, None] * s[None, :, None] * (torch.arange(f.shape[2], device=DEV) <= kc)


def exact(case, seed):
    kind = case["kind"]
    if kind == "ensemble":
        out = []
        for g, u, nu in _members(case, seed):
            u = u.to(torch.complex128)
            for _ in range(case["nsteps"]):
                u = _exact_step(g, dict(eq="hd"), u, None, case["dt"], 4, nu)
            out.append(u)
        return out
    return {"les": _exact_les, "train": _exact_train, "sample": _exact_sample}.get(kind, _exact_solve)(case, seed)
