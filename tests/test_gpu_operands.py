"""Operand preparation of the tensor-core products at the edges of its 8-column
groups and 64 x 64 tiles, from sources that are and are not 16-byte aligned.

The emulated float64 product: digits below 2^-56 of each row's largest entry are
dropped, so per entry 2^-54 K max|A_row| max|B_col| plus the float64 rounding of
the sums, 4 K eps |A||B| with the reference's own. Split-precision products: the
same call on aligned and on shifted copies of the operands gives the same bits."""
import numpy as np
import pytest

from paper_1703_00387_gb300 import binding as B
from paper_1703_00387_gb300 import inputs

pytestmark = pytest.mark.gpu
EPS = np.finfo(float).eps


@pytest.fixture(scope="module")
def ctx():
    c = B.Context(0)
    yield c
    c.close()


def _at(x, shift):
    """x on the device, `shift` doubles past a 16-byte boundary."""
    import torch
    buf = torch.full((x.size + 2,), float("nan"), dtype=torch.float64, device="cuda:0")
    out = buf[shift:shift + x.size].view(*x.shape)
    out.copy_(torch.from_numpy(np.ascontiguousarray(x)))
    return out


@pytest.mark.parametrize("shift", [0, 1])
@pytest.mark.parametrize("M,N,K", [(1, 1, 1), (3, 5, 7), (63, 65, 8), (64, 64, 63), (65, 130, 65), (130, 70, 129),
                                   (20, 200, 2050), (129, 2, 300)])
def test_emulated_product_operand_edges(ctx, M, N, K, shift):
    import torch
    rng = np.random.default_rng(M + N + K)
    a = rng.standard_normal((M, K)) * 2.0 ** rng.integers(-30, 30, (M, 1))
    b = rng.standard_normal((K, N)) * 2.0 ** rng.integers(-30, 30, (1, N))
    a[rng.random(a.shape) < 0.1] = 0.0
    out = torch.full((M, N), float("nan"), dtype=torch.float64, device="cuda:0")
    B.osmps_dgemm_emu(ctx, _at(a, shift), _at(b, shift), out)
    top = np.abs(a).max(1, keepdims=True) * np.abs(b).max(0, keepdims=True)
    bar = 2.0 ** -54 * K * top + 4 * K * EPS * (np.abs(a) @ np.abs(b))
    assert np.all(np.abs(out.cpu().numpy() - a @ b) <= bar)


@pytest.mark.parametrize("prec", ["bf16x3", "tf32x3"])
@pytest.mark.parametrize("chi_l,chi_r", [(64, 64), (63, 65), (70, 9), (129, 130)])
def test_split_operands_do_not_depend_on_alignment(ctx, prec, chi_l, chi_r):
    import torch
    ops = inputs.random_heff_operands(chi_l, 2, 2, chi_r, 5, 5, 5, seed=chi_l)
    env, A, W = inputs.random_env_operands(chi_l, 2, chi_r, 5, 5, 0, seed=chi_r)
    got = []
    for shift in (0, 1):
        t = [_at(x, shift) for x in ops]
        y = torch.full_like(t[4], float("nan"))
        B.osmps_heff_apply(ctx, *t, y, precision=prec)
        e = torch.full((chi_r, 5, chi_r), float("nan"), dtype=torch.float64, device="cuda:0")
        B.osmps_env_update(ctx, 0, _at(env, shift), _at(A, shift), _at(W, shift), e, precision=prec)
        got.append((y.cpu().numpy(), e.cpu().numpy()))
    np.testing.assert_array_equal(got[0][0], got[1][0])
    np.testing.assert_array_equal(got[0][1], got[1][1])
    assert np.isfinite(got[0][0]).all() and np.isfinite(got[0][1]).all()
