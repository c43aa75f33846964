"""Emulated float64 products at the edges of the kernel's work split: a tile's K
blocks shared between blocks of threads, several tiles per block, four and two
diagonals per exact group, partial sums that end at and between whole chunks.

The operands are integers below 2^17 in size, so every slice pair that is left
out is zero and every sum stays below 2^53: the product is exact, and so is the
CPU's. The tolerance is therefore zero."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,N,K", [
    (1, 1, 64),            # one element of one tile, one K block
    (128, 128, 65),        # a second K block of one column
    (127, 129, 257),       # ragged tiles, odd rows: one column per access
    (130, 126, 1024),      # 16 K blocks in shares
    (256, 128, 1087),      # 17 K blocks in shares of unequal length
    (5, 300, 4096),        # eight shares
    (2050, 2040, 64),      # more tiles than SMs
    (1300, 1700, 577),     # the same with ten K blocks
    (3, 2, 131072),        # the longest K of four diagonals to a group
    (3, 130, 131073),      # two diagonals to a group
])
def test_integer_products_are_exact(M, N, K):
    from paper_1703_00387_gb300 import binding as B

    ctx = B.Context(0)
    gen = torch.Generator().manual_seed(M + N + K)
    a = torch.randint(-2**17 + 1, 2**17, (M, K), generator=gen).double()
    b = torch.randint(-2**17 + 1, 2**17, (K, N), generator=gen).double()
    c = torch.full((M, N), float("nan"), dtype=torch.float64, device="cuda")
    B.osmps_dgemm_emu(ctx, a.cuda(), b.cuda(), c)
    assert torch.equal(c.cpu(), a @ b)
