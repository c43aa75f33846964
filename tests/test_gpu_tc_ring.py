"""Ring of K blocks of the split-precision GEMM: two, three or four places (tile
widths 256, 128, 64), each turn round it swaps the places of B's hi and lo tiles.
Lengths of K around whole turns and below one, several tiles to a block of
threads at the last shape.

A tile taken for another is an error of order 1 (hi) or 2^-9 (lo); the products
themselves drop lo * lo, 2^-18 of each term in bf16, and round operands to 2^-17:
below 1e-5 in the 2-norm for random operands, each of two products deep."""
import numpy as np
import pytest

from paper_1703_00387_gb300 import binding as B
from paper_1703_00387_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["bf16x3", "tf32x3"])
@pytest.mark.parametrize("chi_l,chi_r", [(1, 3), (31, 64), (64, 65), (130, 128), (193, 200), (257, 330),
                                         (520, 450), (1300, 1210)])
def test_k_lengths_at_every_width(prec, chi_l, chi_r):
    c = B.Context(0)
    t = [torch.from_numpy(np.ascontiguousarray(x)).cuda()
         for x in inputs.random_heff_operands(chi_l, 2, 2, chi_r, 2, 2, 2, seed=chi_l + chi_r)]
    y, ref = torch.empty_like(t[4]), torch.empty_like(t[4])
    B.osmps_heff_apply(c, *t, ref, precision="fp64")
    B.osmps_heff_apply(c, *t, y, precision=prec)  # tunes both products' classes
    for width in (256, 128, 64):
        for e in c.tuning():
            c.set_tuning(e["key"], width)
        y.fill_(float("nan"))
        B.osmps_heff_apply(c, *t, y, precision=prec)
        assert float((y - ref).norm() / ref.norm()) <= 1e-5
    c.close()
