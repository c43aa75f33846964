"""An Inf or NaN that a block of a W-step kernel meets only in the later ones of
the fibers it walks (more groups of fibers than blocks, the bad row last): it
reaches every output of its row, connected or not, and the other rows keep
their bits."""
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
    """Only output 0 of the last index is connected, and a few entries more."""
    V = np.zeros_like(W)
    V[:, 0, 0, 0] = 1.0
    V[0, 1, 0, 0] = 0.5
    return V


# both W-steps in one pass: 16-byte and scalar fibers; two passes (d1 != d2)
@pytest.mark.parametrize("shape,prec", [
    ((300, 2, 2, 300, 5, 5, 5), "fp64"),
    ((301, 2, 2, 257, 5, 5, 5), "fp64"),
    ((200, 3, 3, 200, 14, 14, 14), "tf32x3"),
    ((300, 2, 3, 300, 4, 4, 4), "fp64"),
    ((300, 2, 3, 300, 4, 4, 4), "bf16x3"),
], ids=str)
@pytest.mark.parametrize("bad", [np.inf, np.nan])
def test_product(ctx, shape, prec, bad):
    import torch
    Lh, W1, W2, Rh, th = inputs.random_heff_operands(*shape, seed=5)
    t = [torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in (Lh, _sparse(W1), _sparse(W2), Rh, th)]
    ref, y = torch.zeros_like(t[4]), torch.zeros_like(t[4])
    B.osmps_heff_apply(ctx, *t, ref, precision=prec)
    assert torch.isfinite(ref).all()
    t[0][-1, 1, 2] = bad  # the last bra row only
    B.osmps_heff_apply(ctx, *t, y, precision=prec)
    assert torch.isnan(y[-1]).all()
    assert torch.equal(y[:-1], ref[:-1])


@pytest.mark.parametrize("chi_l,d,chi_r,w", [(400, 2, 400, 5), (401, 3, 301, 7)])
def test_right_update(ctx, chi_l, d, chi_r, w):
    import torch
    env, A, W = inputs.random_env_operands(chi_l, d, chi_r, w, w, 1, seed=6)
    t = [torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in (env, A, _sparse(W))]
    ref, out = (torch.zeros(chi_l, w, chi_l, dtype=torch.float64, device="cuda") for _ in range(2))
    B.osmps_env_update(ctx, 1, *t, ref, precision="fp64")
    t[1][-1, 0, 5] = float("nan")
    B.osmps_env_update(ctx, 1, *t, out, precision="fp64")
    assert torch.isnan(out[-1]).all() and torch.isnan(out[:, :, -1]).all()
    assert torch.equal(out[:-1, :, :-1], ref[:-1, :, :-1])
