"""The W-steps of H_eff.theta at the shapes where their kernels change: fibers
that fill no block, one and several threads per column buffer (d = 2 ... 5,
blocks of 128, 64 and 32 threads), dense MPO tensors, MPO tensors with empty
rows and columns, d1 != d2 and d = 6 (two separate passes), an input side too
long for shared memory. Bars per
entry, on the product of absolute values: a bf16 pair leaves 2^-18 |x| and the
dropped lo.lo term 2^-18, three such terms in each of two products, so 2^-15
with the float32 sums; tf32 pairs 2^-22 each, so 2^-19; float64 sums 4 eps per
term.
"""
import numpy as np
import pytest

from oracle import dmrg as odmrg
from paper_1703_00387_gb300 import binding as B
from paper_1703_00387_gb300 import inputs

pytestmark = pytest.mark.gpu
SHAPES = [(1, 2, 2, 1, 1, 1, 1), (3, 2, 2, 5, 4, 4, 4), (33, 2, 2, 31, 6, 7, 5), (20, 3, 3, 17, 14, 14, 14),
          (9, 4, 4, 21, 9, 8, 7), (12, 5, 5, 13, 4, 4, 4), (7, 5, 5, 9, 12, 12, 12), (10, 6, 6, 11, 3, 3, 3),
          (10, 2, 3, 11, 4, 5, 3), (4, 2, 2, 6, 400, 2, 2), (40, 2, 2, 1, 10, 10, 10)]


@pytest.fixture(scope="module")
def ctx():
    c = B.Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("zeros", [0.0, 0.8])
@pytest.mark.parametrize("prec,bar", [("fp64", None), ("bf16x3", 2.0 ** -15), ("tf32x3", 2.0 ** -19)])
@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "x".join(map(str, s)))
def test_wsteps_shapes(ctx, shape, prec, bar, zeros):
    import torch
    Lh, W1, W2, Rh, th = inputs.random_heff_operands(*shape, seed=sum(shape))
    if zeros:
        rng = np.random.default_rng(1)
        W1, W2 = (w * (rng.random(w.shape) >= zeros) for w in (W1, W2))
        W1[..., 0] = 1.0  # something is left
        W2[0] = 1.0
    ref = odmrg.heff_apply(Lh, W1, W2, Rh, th)
    t = [torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in (Lh, W1, W2, Rh, th)]
    y = torch.full_like(t[4], float("nan"))
    B.osmps_heff_apply(ctx, *t, y, precision=prec)
    chi_l, d1, d2, chi_r, wl, wm, wr = shape
    bar = bar or 4 * (chi_l + d1 * wl + d2 * wm + wr * chi_r) * np.finfo(float).eps
    mag = odmrg.heff_apply(*(np.abs(x) for x in (Lh, W1, W2, Rh, th)))
    assert np.all(np.abs(y.cpu().numpy() - ref) <= bar * mag)
