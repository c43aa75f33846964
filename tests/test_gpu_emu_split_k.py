"""Emulated float64 products whose K blocks are shared between blocks of
threads: the shares are added as exact integers, so an entry has the same bits
as in a product of enough tiles to need no shares (the same operands beside
more columns). Tolerance: none."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,N,K", [
    (128, 128, 1024),     # shares of equal length, one tile
    (130, 126, 2000),     # ragged tiles and K
    (1, 3, 4096),
    (300, 257, 1087),     # 17 K blocks
    (512, 512, 2048),
    (129, 66, 640),
])
@pytest.mark.parametrize("scale", [1.0, 1e-200])  # (tiny: scales far from 1)
def test_shares_leave_the_bits(M, N, K, scale):
    from paper_1703_00387_gb300 import binding as B

    ctx = B.Context(0)
    tiles_m = -(-M // 128)
    wide = 128 * (320 // tiles_m + 1)  # past two tiles per SM: no shares
    gen = torch.Generator(device="cuda").manual_seed(M + N + K)
    a = torch.randn(M, K, generator=gen, dtype=torch.float64, device="cuda") * scale
    b = torch.randn(K, N, generator=gen, dtype=torch.float64, device="cuda")
    bw = torch.zeros(K, wide, dtype=torch.float64, device="cuda")
    bw[:, :N] = b
    c = torch.full((M, N), float("nan"), dtype=torch.float64, device="cuda")
    cw = torch.full((M, wide), float("nan"), dtype=torch.float64, device="cuda")
    B.osmps_dgemm_emu(ctx, a, b, c)
    B.osmps_dgemm_emu(ctx, a, bw, cw)
    assert torch.equal(c, cw[:, :N])
    assert (cw[:, N:] == 0).all()
    ctx.close()
