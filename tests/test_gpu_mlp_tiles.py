"""The MLP kernels at the edges of their tiles (16 samples a warp tile, 128 a
chunk) and of the loss sum's FP32 range, against the FP64 oracle fed the same
BF16 operand rounding."""

import numpy as np
import pytest

from oracle import les

from .test_gpu_mlp import ORDER, _case, pack, relerr, unpack

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

EDGES = [1, 15, 16, 17, 33, 127, 128, 129, 257]
# One operand whose FP32 and FP64 values round to different BF16 neighbours
# moves an output by up to 2^-9 |h w3| ~ 2.5e-4 of order-one residuals: 1e-3 of
# a loss over few samples, and within the 2e-2 of the gradients.
LOSS_TOL = 1e-3
GRAD_TOL = 2e-2


@pytest.fixture(scope="module")
def ps():
    import __graft_entry__
    __graft_entry__.build()
    from paper_1808_01309_gb300 import ps as _ps
    return _ps


def _cuda(*arrays):
    return [torch.from_numpy(np.ascontiguousarray(a)).to("cuda") for a in arrays]


@pytest.mark.parametrize("B", EDGES)
def test_forward_and_backward_at_tile_edges(ps, B):
    p, X, T = _case(20 + B, B)
    P, Xd, Td = _cuda(pack(p), X, T)
    Y = torch.full((B + 1, 6), 7.0, device="cuda")
    ps.ps_mlp_forward(P, Xd, Y, B)
    y_ref, cache = les.mlp_forward(p, X.astype(np.float64), rnd=les.bf16_round)
    assert relerr(Y[:B].cpu().numpy(), y_ref) < 2e-3
    assert bool((Y[B] == 7.0).all())  # nothing written past the last sample
    grad = torch.empty(ps.MLP_NPARAM, device="cuda")
    loss = torch.empty(1, device="cuda", dtype=torch.float64)
    ps.ps_mlp_grad(P, Xd, Td, B, grad, loss)
    L, g = les.mse_and_grads(p, X.astype(np.float64), T.astype(np.float64), rnd=les.bf16_round)
    assert abs(float(loss) - L) < LOSS_TOL * L
    got = unpack(grad.cpu().numpy())
    assert all(relerr(got[k], g[k]) < GRAD_TOL for k in ORDER)
    # backpropagation of given output deltas adds to the gradient
    ps.ps_mlp_backward(P, Xd, Td, B, grad)
    g2 = les._backward(p, cache, T.astype(np.float64), les.bf16_round)
    got = unpack(grad.cpu().numpy())
    assert all(relerr(got[k], g[k] + g2[k]) < GRAD_TOL for k in ORDER)


@pytest.mark.parametrize("B", EDGES)
def test_tensor_basis_fit_at_tile_edges(ps, B):
    p, X, T = _case(40 + B, B)
    A = np.random.default_rng(B).standard_normal((B, 9)).astype(np.float32)
    P, Xd, Ad, Td = _cuda(pack(p), X, A, T)
    grad = torch.empty(ps.MLP_NPARAM, device="cuda")
    loss = torch.empty(1, device="cuda", dtype=torch.float64)
    ps.ps_mlp_grad_tb(P, Xd, Ad, Td, B, 1.7, 0.3, grad, loss)
    Bas = les.tensor_basis(A.astype(np.float64).T.reshape(3, 3, B), 1.7).transpose(2, 1, 0)
    L, g = les.mse_and_grads_tb(p, X.astype(np.float64), Bas, T.astype(np.float64) / 0.3, rnd=les.bf16_round)
    assert abs(float(loss) - L) < LOSS_TOL * L
    got = unpack(grad.cpu().numpy())
    assert all(relerr(got[k], g[k]) < GRAD_TOL for k in ORDER)


@pytest.mark.parametrize("size", [1e-18, 1e-3, 1e12, 1e17, 1e30])
def test_loss_of_residuals_beyond_the_fp32_range_of_their_squares(ps, size):
    p, X, T = _case(3, 200)
    for k in ("W3", "b3"):
        p[k] = p[k] * 0.0  # outputs zero: the residuals are the targets
    T = (T * size).astype(np.float32)
    P, Xd, Td = _cuda(pack(p), X, T)
    grad = torch.empty(ps.MLP_NPARAM, device="cuda")
    loss = torch.empty(1, device="cuda", dtype=torch.float64)
    ps.ps_mlp_grad(P, Xd, Td, 200, grad, loss)
    L = float(np.mean(T.astype(np.float64) ** 2))
    # 1200 sums of 48-bit pairs
    assert abs(float(loss) - L) < 1e-12 * L
