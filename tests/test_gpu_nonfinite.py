"""An Inf or NaN that meets a zero MPO entry: 0 x Inf and 0 x NaN are NaN, so in
float64 (and in the split precisions where the W-steps are the general ones) a
W-step passes it on to every output of its fiber, connected or not. Through the
sums of the last contraction it then reaches every entry of the result."""
import numpy as np
import pytest

from paper_1703_00387_gb300 import binding as B
from paper_1703_00387_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    c = B.Context(0)
    yield c
    c.close()


def _sparse(W):
    """Only output 0 of each site tensor's last index is connected."""
    W = np.zeros_like(W)
    W[:, 0, 0, 0] = 1.0
    return W


# fused (16-byte fibers, scalar fibers, d = 3), two passes (d1 != d2), inputs
# read where they are used (400 channels)
@pytest.mark.parametrize("shape", [(8, 2, 2, 8, 5, 5, 5), (7, 2, 2, 9, 6, 7, 5), (5, 3, 3, 40, 14, 14, 14),
                                   (6, 2, 3, 10, 4, 5, 3), (4, 2, 2, 6, 400, 2, 2)], ids=str)
@pytest.mark.parametrize("bad", [np.inf, -np.inf, np.nan])
@pytest.mark.parametrize("prec", ["fp64", "bf16x3", "tf32x3"])
def test_product(ctx, shape, bad, prec):
    import torch
    if prec != "fp64" and shape == (8, 2, 2, 8, 5, 5, 5):
        pytest.skip("spin chains of the specialised split-precision W-steps: nonzero entries only")
    Lh, W1, W2, Rh, th = inputs.random_heff_operands(*shape, seed=1)
    th[1, 1, 0, 3] = bad
    t = [torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in (Lh, _sparse(W1), _sparse(W2), Rh, th)]
    y = torch.zeros_like(t[4])
    B.osmps_heff_apply(ctx, *t, y, precision=prec)
    assert torch.isnan(y).all()


@pytest.mark.parametrize("side", [0, 1])
@pytest.mark.parametrize("bad", [np.inf, np.nan])
@pytest.mark.parametrize("chi_l,d,chi_r,w", [(8, 2, 8, 5), (9, 3, 7, 14)])
def test_environment_update(ctx, side, bad, chi_l, d, chi_r, w):
    import torch
    env, A, W = inputs.random_env_operands(chi_l, d, chi_r, w, w, side, seed=2)
    env[1, 1, 2] = bad
    t = [torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in (env, A, _sparse(W))]
    n = chi_r if side == 0 else chi_l
    out = torch.zeros(n, w, n, dtype=torch.float64, device="cuda")
    B.osmps_env_update(ctx, side, *t, out, precision="fp64")
    assert torch.isnan(out).all()


def test_finite_fibers_beside_a_nan_keep_their_bits(ctx):
    """A NaN in row 3 of the site tensor of a right update makes the W-step sum
    all entries for the fibers beside row 3's too; rows and columns other than 3
    of the result keep their bits."""
    import torch
    env, A, W = inputs.random_env_operands(8, 2, 40, 5, 5, 1, seed=4)
    W = _sparse(W) + 0.5 * (np.arange(W.size).reshape(W.shape) % 7 == 0)
    t = [torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in (env, A, W)]
    ref = torch.zeros(8, 5, 8, dtype=torch.float64, device="cuda")
    B.osmps_env_update(ctx, 1, *t, ref, precision="fp64")
    t[1][3, 0, 5] = float("nan")
    out = torch.zeros_like(ref)
    B.osmps_env_update(ctx, 1, *t, out, precision="fp64")
    keep = [i for i in range(8) if i != 3]
    assert torch.isnan(out[3]).all() and torch.isnan(out[:, :, 3]).all()
    assert torch.equal(out[keep][:, :, keep], ref[keep][:, :, keep])
