"""A sample with a NaN or an infinity among its inputs changes no other sample's
output: inference runs 16-sample tiles through one warp, and every other row of
the batch keeps its value bit for bit."""

import math

import numpy as np
import pytest

from .test_gpu_mlp import _case, pack

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

B = 33  # two full tiles and one sample


@pytest.fixture(scope="module")
def ps():
    import __graft_entry__
    __graft_entry__.build()
    from paper_1808_01309_gb300 import ps as _ps
    return _ps


def _forward(ps, P, X):
    Y = torch.full((B, 6), 7.0, device="cuda")
    ps.ps_mlp_forward(P, torch.from_numpy(X).to("cuda"), Y, B)
    return Y.cpu().numpy()


@pytest.mark.parametrize("row", [0, 3, 11, 15, 24, 32])
@pytest.mark.parametrize("bad", [math.nan, math.inf, -math.inf])
def test_other_samples_keep_their_outputs(ps, bad, row):
    p, X, _ = _case(51, B)
    P = torch.from_numpy(pack(p)).to("cuda")
    want = _forward(ps, P, X)
    assert np.isfinite(want).all()
    X[row, 2] = bad
    got = _forward(ps, P, X)
    rest = np.arange(B) != row
    assert np.array_equal(got[rest], want[rest])
    if math.isnan(bad):
        assert np.isnan(got[row]).all()
