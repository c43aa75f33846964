"""Every slice pair of the emulated float64 product by itself: A holds digits of
slice a only and B of slice b only (a + b <= 7), so the product is that pair's
one integer sum at its weight, and any slice taken from a wrong place of the
ring, released early or left out of a partial sum shows. Each row's (column's)
exponent is pinned by a large entry at a K index where the other operand is
zero. Digits are below 64 in size and the integer sums below 2^53, so expected
values and float64 sums of the reference are exact. Tolerance: none."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu
PAIRS = [(a, b) for a in range(8) for b in range(8 - a)]


@pytest.fixture(scope="module")
def ctx():
    from paper_1703_00387_gb300 import binding as B

    c = B.Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("M,N,K", [
    (130, 126, 70),       # two K blocks, ragged tiles
    (130, 126, 1090),     # K blocks in shares
    (1300, 1700, 577),    # several tiles per block of threads
    (1300, 2300, 2112),   # the same with several partial sums per diagonal
    (3, 5, 131130),       # two diagonals to a group
])
def test_each_pair_is_exact(ctx, M, N, K):
    from paper_1703_00387_gb300 import binding as B

    gen = torch.Generator(device="cuda").manual_seed(M + K)
    dev = dict(dtype=torch.float64, device="cuda")
    sa, sb = (torch.from_numpy(np.ldexp(1.0, np.random.default_rng(n).integers(-40, 40, n))).cuda() for n in (M, N))
    sa, sb = sa[:, None], sb[None, :]  # exact powers of two
    da = torch.randint(-63, 64, (M, K), generator=gen, device="cuda").double()
    db = torch.randint(-63, 64, (K, N), generator=gen, device="cuda").double()
    pin_a, pin_b = K // 3, K - 1  # A large where B is zero, and the other way round
    for m, k in ((da, pin_a), (da, pin_b)):
        m[:, k] = 0.0
    for m, k in ((db, pin_a), (db, pin_b)):
        m[k, :] = 0.0
    sums = da @ db
    out = torch.empty(M, N, **dev)
    for a, b in PAIRS:
        A, Bm = da * 2.0 ** (-7 * (a + 1)), db * 2.0 ** (-7 * (b + 1))
        A[:, pin_a] = 0.75
        Bm[pin_b, :] = 0.75
        out.fill_(float("nan"))
        B.osmps_dgemm_emu(ctx, A * sa, Bm * sb, out)
        assert torch.equal(out, sums * 2.0 ** (-7 * (a + b + 2)) * sa * sb), (a, b)
