"""Both words of the float64 operand splits (bf16 and tf32 pairs, formed with
integer operations) equal the hardware conversions bit for bit: random values
over the float32 range and beyond, values that are exactly representable (lo =
0), hi rounded up across a power of two, lo exactly halfway between neighbours
(both parities and signs), lo at and under the smallest normal number, exponents
at both ends of the integer path, zeros, infinities and NaN."""
import numpy as np
import pytest

from paper_1703_00387_gb300 import binding as B

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    c = B.Context(0)
    yield c
    c.close()


def _edges(bits):
    """bits: significant bits of one word (8 for bf16, 11 for tf32)."""
    rng = np.random.default_rng(bits)
    one = []
    u = 2.0 ** (1 - bits)  # spacing of the words in [1, 2)
    for hi in (1.0, 1.0 + u, 1.0 + 2 * u, 2.0 - u, 1.5):
        for lo in (0.0, u / 2, u / 4, u / 8, u / 2 - 2.0 ** -40, u / 4 + 2.0 ** -45, 2.0 ** -52, 2.0 ** -51):
            for sgn in (1.0, -1.0):
                one.append(hi + sgn * lo)
        # lo halfway between two of its own words: m + half a unit, at several sizes
        for e in (2, 3, 5, 9):
            for m in (2 ** (bits - 1), 2 ** (bits - 1) + 1, 2 ** bits - 1):
                lo = (m + 0.5) * u * 2.0 ** -(bits - 1 + e)
                one += [hi + lo, hi - lo, hi + lo * (1 + 2.0 ** -20)]
        one += [hi + u / 2 * (1 + 2.0 ** -30), hi + u / 2 * (1 - 2.0 ** -30)]
    one = np.array(one + list(rng.uniform(1.0, 2.0, 200)))
    scales = np.concatenate([np.arange(-160, -100), np.arange(-20, 20, 7), np.arange(118, 130)]).astype(float)
    x = np.ldexp(one[None, :], scales.astype(int)[:, None]).ravel()
    tiny = float(np.finfo(np.float32).tiny)
    special = [0.0, -0.0, np.inf, -np.inf, np.nan, 1e-300, 1e300, 3.3e38, 3.4028235e38, 3.5e38, tiny, tiny / 2, tiny / 3,
               5e-324, 1.7e308]
    return np.concatenate([x, -x, np.array(special), -np.array(special)])


@pytest.mark.parametrize("prec,bits", [("bf16x3", 8), ("tf32x3", 11)])
def test_split_words(ctx, prec, bits):
    rng = np.random.default_rng(0)
    n = 1 << 21
    with np.errstate(over="ignore", under="ignore"):
        x = np.ldexp(rng.uniform(1.0, 2.0, n), rng.integers(-170, 135, n)) * rng.choice([-1.0, 1.0], n)
        short = np.ldexp(rng.integers(1, 2 ** 20, n).astype(float), rng.integers(-140, 100, n))  # many ties
        x = np.concatenate([x, short, _edges(bits)])
    got, ref = B.osmps_selftest_split(ctx, torch.from_numpy(x).cuda(), prec)
    got, ref = got.cpu().numpy(), ref.cpu().numpy()
    bad = np.nonzero((got != ref).any(1))[0]
    assert bad.size == 0, [(x[i].hex(), got[i].tolist(), ref[i].tolist()) for i in bad[:5]]


def test_split_refuses(ctx):
    x = torch.ones(4, dtype=torch.float64, device="cuda")
    for prec in ("fp64", "fp64emu", 9):
        with pytest.raises(B.OsmpsError) as e:
            B.osmps_selftest_split(ctx, x, prec)
        assert e.value.status == B.EINVAL
